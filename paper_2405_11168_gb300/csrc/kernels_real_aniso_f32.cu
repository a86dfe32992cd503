// Real-space pass, float, anisotropic phases.
#include "kernels_real.cuh"
HS_INSTANTIATE_REAL(float, false, RealAniso<float>)
