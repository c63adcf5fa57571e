// Stage kernels of two-dimensional boxes for the fp64 form.
#define MHD_UNIT_PREC P_FP64
#define MHD_UNIT_FN(name) name##_fp64
#define MHD_TILES(X) X(16, 8) X(24, 8) X(8, 8)
#include "stage2d_unit.cuh"
