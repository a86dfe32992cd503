// FP32 column passes (wider tile: 16 complex = 128 B).
#include "kernels_impl.cuh"
HS_INSTANTIATE_COLS(float, 16)
