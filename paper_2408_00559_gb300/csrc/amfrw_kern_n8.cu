// Solver kernels for N = 8 axes (7 forward rate(s) and V).
#include "amfrw_kernels.cuh"
AMFRW_INSTANTIATE(8)
