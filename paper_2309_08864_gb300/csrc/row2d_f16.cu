// row2d_f16.cu -- 2D temporal-blocking kernels for f16 storage.
#define STORAGE_T __half
#define STORAGE_F64 0
#define ROW_LAUNCH_FN launch_row2d_f16
#define ROW_OCC_FN occupancy_row2d_f16
#include "row2d_inst.inc"
