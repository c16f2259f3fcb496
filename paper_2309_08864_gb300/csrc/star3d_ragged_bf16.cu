// star3d_ragged_bf16.cu -- 3D star temporal-blocking kernels for bf16 storage, rows of any length.
#include <cstring>
#define STORAGE_T __nv_bfloat16
#define STAGE_RAGGED 1
#define STAR_LAUNCH_FN launch_star3d_ragged_bf16
#define STAR_OCC_FN occupancy_star3d_ragged_bf16
#include "star3d_inst.inc"
