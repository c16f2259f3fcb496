// row2d_f32.cu -- 2D temporal-blocking kernels for f32 storage.
#define STORAGE_T float
#define STORAGE_F64 0
#define ROW_LAUNCH_FN launch_row2d_f32
#define ROW_OCC_FN occupancy_row2d_f32
#include "row2d_inst.inc"
