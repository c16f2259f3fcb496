// star3d_ragged_f32.cu -- 3D star temporal-blocking kernels for f32 storage, rows of any length.
#include <cstring>
#define STORAGE_T float
#define STAGE_RAGGED 1
#define STAR_LAUNCH_FN launch_star3d_ragged_f32
#define STAR_OCC_FN occupancy_star3d_ragged_f32
#include "star3d_inst.inc"
