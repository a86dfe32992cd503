// FP64 column passes (wider tile: 8 complex = 128 B).
#include "kernels_impl.cuh"
HS_INSTANTIATE_COLS(double, 8)
