// Real-space pass, double, anisotropic phases.
#include "kernels_real.cuh"
HS_INSTANTIATE_REAL(double, false, RealAniso<double>)
