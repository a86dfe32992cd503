// Real-space pass, double, isotropic phases.
#include "kernels_real.cuh"
HS_INSTANTIATE_REAL(double, true, RealIso<double>)
