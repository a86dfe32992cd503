// Definitions of the real-space pass's launchers (launch.h); included once per precision and law.
#pragma once
#include "launch_util.cuh"
#include "real.cuh"

namespace hs {

template <typename T, int TY, class MAT, int MODE, int XP, int NT, int OPT, bool BATCH>
static cudaError_t real_one(const MarchArgs<T>& a, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  auto k = k_real<T, TY, MAT, MODE, XP, NT, OPT, BATCH>;
  if (nthr > NT || (XP > 0 && occ == nullptr && a.xp != XP)) return cudaErrorInvalidValue;
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  if (occ != nullptr) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, nthr, smem);
  if constexpr ((OPT & REAL_SPLIT) != 0) {
    if (!a.bulk || nthr != real_threads(true, TY, a.n1)) return cudaErrorInvalidValue;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = dim3((unsigned)nthr);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a, MAT{a.mat});
  } else {
    k<<<g, nthr, smem, s>>>(a, MAT{a.mat});
    return cudaGetLastError();
  }
}

// batched launches (zstride != 0) run the force pass without an eigenstrain only
template <typename T, int TY, class MAT, int MODE, int XP, int NT, int OPT>
static cudaError_t real_batch(const MarchArgs<T>& a, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  if (a.zstride != 0) {
    if constexpr (MODE == MODE_FORCE && !(OPT & REAL_EIGEN))
      return real_one<T, TY, MAT, MODE, XP, NT, OPT, true>(a, g, nthr, smem, s, occ);
    else return cudaErrorInvalidValue;
  }
  return real_one<T, TY, MAT, MODE, XP, NT, OPT, false>(a, g, nthr, smem, s, occ);
}

// A launch has a source (correction solves, FP32 force passes only) or an eigenstress, or neither.
template <typename T, int TY, class MAT, int MODE, int XP, int NT, int B = 0>
static cudaError_t real_opt(const MarchArgs<T>& a, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  if (a.src != nullptr) {
    if constexpr (sizeof(T) == 4 && MODE == MODE_FORCE) {
      if (a.sig0 != nullptr) return cudaErrorInvalidValue;
      return real_batch<T, TY, MAT, MODE, XP, NT, B | REAL_SRC>(a, g, nthr, smem, s, occ);
    } else {
      return cudaErrorInvalidValue;
    }
  }
  if (a.sig0 != nullptr) return real_batch<T, TY, MAT, MODE, XP, NT, B | REAL_EIGEN>(a, g, nthr, smem, s, occ);
  return real_batch<T, TY, MAT, MODE, XP, NT, B>(a, g, nthr, smem, s, occ);
}

template <typename T, int TY, class MAT, int MODE>
static cudaError_t real_xp(const MarchArgs<T>& a, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  if constexpr (sizeof(T) == 8) {
    if constexpr (TY == 8) {
      if (!real_rows_fit(true, TY, a.n1)) return cudaErrorInvalidValue;
      if (real_split(true, TY, a.n1)) return real_opt<T, TY, MAT, MODE, 0, 256, REAL_SPLIT>(a, g, nthr, smem, s, occ);
    }
    if (nthr <= 256) return real_opt<T, TY, MAT, MODE, 0, 256>(a, g, nthr, smem, s, occ);
    if constexpr (TY < 8) return real_opt<T, TY, MAT, MODE, 0, 512>(a, g, nthr, smem, s, occ);
    else return cudaErrorInvalidValue;
  } else if constexpr (TY == 4 && MODE == MODE_FORCE) {
    switch (real_pitch_class(false, TY, MODE, a.n1)) {
#define HS_CASE(P)                                                                                     \
  case P:                                                                                              \
    return a.bulk || occ != nullptr ? real_opt<T, TY, MAT, MODE, P, P, REAL_BULK>(a, g, nthr, smem, s, occ) \
                                    : real_opt<T, TY, MAT, MODE, P, P, 0>(a, g, nthr, smem, s, occ);
      HS_CASE(64)
      HS_CASE(128)
      HS_CASE(256)
      HS_CASE(512)
#undef HS_CASE
      default: return cudaErrorInvalidValue;
    }
  } else {
    return real_opt<T, TY, MAT, MODE, 0, 512>(a, g, nthr, smem, s, occ);
  }
}

template <typename T, int TY, class MAT>
static cudaError_t real_mode(const MarchArgs<T>& a, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  switch (mode) {
    case MODE_FORCE: return real_xp<T, TY, MAT, MODE_FORCE>(a, g, nthr, smem, s, occ);
    case MODE_FIELDS: return real_xp<T, TY, MAT, MODE_FIELDS>(a, g, nthr, smem, s, occ);
    case MODE_FORCE_FIELDS:  // last FP64 residual sweep of a refined solve
      if constexpr (sizeof(T) == 8) return real_xp<T, TY, MAT, MODE_FORCE_FIELDS>(a, g, nthr, smem, s, occ);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, class MAT>
static cudaError_t real_ty(const MarchArgs<T>& a, int ty, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s,
                           int* occ) {
  switch (ty) {
    case 2: return real_mode<T, 2, MAT>(a, mode, g, nthr, smem, s, occ);
    case 4: return real_mode<T, 4, MAT>(a, mode, g, nthr, smem, s, occ);
    case 8: return real_mode<T, 8, MAT>(a, mode, g, nthr, smem, s, occ);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace hs

#define HS_INSTANTIATE_REAL(T, ISO, MAT)                                                                  \
  namespace hs {                                                                                         \
  template <>                                                                                            \
  cudaError_t launch_real_law<T, ISO>(const MarchArgs<T>& a, int ty, int mode, dim3 grid, int nthr, size_t smem, \
                                      cudaStream_t s, int* occ) {                                        \
    if (occ == nullptr) {                                                                                \
      if (a.ids == nullptr || a.mat == nullptr || a.st == nullptr || a.partials == nullptr || a.ureal == nullptr) \
        return cudaErrorInvalidValue;                                                                    \
      if ((mode == MODE_FIELDS || mode == MODE_FORCE_FIELDS) && (a.eps_out == nullptr || a.sig_out == nullptr)) \
        return cudaErrorInvalidValue;                                                                    \
    }                                                                                                    \
    return real_ty<T, MAT>(a, ty, mode, grid, nthr, smem, s, occ);                                       \
  }                                                                                                      \
  }
