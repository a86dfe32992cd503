// FP32 persistent column passes.
#include "kernels_impl.cuh"
HS_INSTANTIATE_COLP(float, 8)
