// star3d_f16.cu -- 3D star temporal-blocking kernels for f16 storage.
#include <cstring>
#define STORAGE_T __half
#define STAGE_RAGGED 0
#define STAR_LAUNCH_FN launch_star3d_f16
#define STAR_OCC_FN occupancy_star3d_f16
#include "star3d_inst.inc"
