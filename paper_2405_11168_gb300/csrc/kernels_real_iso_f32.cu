// Real-space pass, float, isotropic phases.
#include "kernels_real.cuh"
HS_INSTANTIATE_REAL(float, true, RealIso<float>)
