// FP64 row passes.
#include "kernels_impl.cuh"
HS_INSTANTIATE_ROWS(double)
