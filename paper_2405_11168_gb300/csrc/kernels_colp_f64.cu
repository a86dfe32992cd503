// FP64 persistent column passes.
#include "kernels_impl.cuh"
HS_INSTANTIATE_COLP(double, 4)
