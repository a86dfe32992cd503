// FP32 fused x pass and state import / export.
#include "kernels_impl.cuh"
HS_INSTANTIATE(float)
