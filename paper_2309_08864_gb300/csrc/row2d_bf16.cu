// row2d_bf16.cu -- 2D temporal-blocking kernels for bf16 storage.
#define STORAGE_T __nv_bfloat16
#define STORAGE_F64 0
#define ROW_LAUNCH_FN launch_row2d_bf16
#define ROW_OCC_FN occupancy_row2d_bf16
#include "row2d_inst.inc"
