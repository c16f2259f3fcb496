// row2d_f64.cu -- 2D temporal-blocking kernels for f64 storage.
#define STORAGE_T double
#define STORAGE_F64 1
#define ROW_LAUNCH_FN launch_row2d_f64
#define ROW_OCC_FN occupancy_row2d_f64
#include "row2d_inst.inc"
