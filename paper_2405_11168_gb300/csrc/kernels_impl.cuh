// Definitions of the launchers in launch.h; included once per precision.
#pragma once
#include <string.h>

#include "launch_util.cuh"

namespace hs {

template <typename T, int TY, class MAT, int MODE>
static cudaError_t march_one(const MarchArgs<T>& a, const MAT& m, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  auto k = k_march<T, TY, MAT, MODE>;
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<g, nthr, smem, s>>>(a, m);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t march_ty(const MarchArgs<T>& a, bool iso, int mode, dim3 g, int nthr, size_t smem,
                            cudaStream_t s) {
  const MatIso<T> mi{a.mat};
  const MatAniso<T> ma{a.mat};
  switch (mode) {
    case MODE_EMIT: return march_one<T, TY, MatIso<T>, MODE_EMIT>(a, mi, g, nthr, smem, s);
    case MODE_FORCE:
      return iso ? march_one<T, TY, MatIso<T>, MODE_FORCE>(a, mi, g, nthr, smem, s)
                 : march_one<T, TY, MatAniso<T>, MODE_FORCE>(a, ma, g, nthr, smem, s);
    case MODE_FIELDS:
      return iso ? march_one<T, TY, MatIso<T>, MODE_FIELDS>(a, mi, g, nthr, smem, s)
                 : march_one<T, TY, MatAniso<T>, MODE_FIELDS>(a, ma, g, nthr, smem, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int CT, int MODE, int LF = 0, int NT = 0>
static cudaError_t col_one(const ColArgs<T>& a, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  auto k = k_col<T, CT, MODE, LF, NT>;
  if constexpr (MODE != COL_Z_INV_STATE && LF > 0) {
    if (a.tma && !(MODE == COL_Z_GREEN && a.state_smem)) k = k_col<T, CT, MODE, LF, NT, true>;
  }
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  return launch_pass(k, a, pass_dependent<T>(a.zstride, (size_t)a.n1 * a.n2 * a.n3), g, nthr, smem, s);
}

template <typename T, int CT, int LF = 0, int NT = 0>
static cudaError_t col_ct(const ColArgs<T>& a, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  switch (mode) {
    case COL_Y_FWD: return col_one<T, CT, COL_Y_FWD, LF, NT>(a, g, nthr, smem, s);
    case COL_Y_INV: return col_one<T, CT, COL_Y_INV, LF, NT>(a, g, nthr, smem, s);
    case COL_Z_GREEN: return col_one<T, CT, COL_Z_GREEN, LF, NT>(a, g, nthr, smem, s);
    case COL_Z_INV_STATE: return col_one<T, CT, COL_Z_INV_STATE, LF, NT>(a, g, nthr, smem, s);
    default: return cudaErrorInvalidValue;
  }
}

// transformed length of a column pass
template <typename T> static int col_length(const ColArgs<T>& a, int mode) {
  return (mode == COL_Y_FWD || mode == COL_Y_INV) ? a.n2 : a.n3;
}

// The FP32-only lengths (kernels_more_*_f32.cu); *ran: one of them with its block.
template <int CT>
static cudaError_t col_dispatch_f32(const ColArgs<float>& a, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s,
                                    bool* ran) {
  const int L = col_length(a, mode);
  *ran = fft_fixed_length(L, false) && nthr == col_block(fft_threads<ColPlan>(L, false), 3 * CT, false);
  if (!*ran) return cudaSuccess;
  return launch_col_more(a, mode, L, g, nthr, smem, s);
}

// compile-time variants for the default tile and block size at the lengths that have a plan
template <typename T, int CT>
static cudaError_t col_dispatch(const ColArgs<T>& a, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  switch (col_length(a, mode)) {
#define HS_CASE(LEN)                                                                        \
  case LEN: {                                                                               \
    constexpr int NT = col_block(ColPlan<LEN>::T, 3 * CT, sizeof(T) == 8);                \
    if (nthr == NT) return col_ct<T, CT, LEN, NT>(a, mode, g, nthr, smem, s);               \
    break;                                                                                  \
  }
    HS_FIXED_LENGTHS(HS_CASE)
#undef HS_CASE
  }
  if constexpr (sizeof(T) == 4) {
    bool ran = false;
    const cudaError_t e = col_dispatch_f32<CT>(a, mode, g, nthr, smem, s, &ran);
    if (ran) return e;
  }
  if (plan_ext(a.plan)) return launch_col_ext<T>(a, mode, CT, g, nthr, smem, s);
  return col_ct<T, CT>(a, mode, g, nthr, smem, s);
}

template <typename T, int CT, int MODE, int LF, int NT>
static cudaError_t colp_one(const ColArgs<T>& a, dim3 g, size_t smem, cudaStream_t s, int* occ) {
  auto k = k_colp<T, CT, MODE, LF, NT>;
  if (a.tma) k = k_colp<T, CT, MODE, LF, NT, true>;
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  if (occ != nullptr) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, NT, smem);
  return launch_pass(k, a, pass_dependent<T>(a.zstride, (size_t)a.n1 * a.n2 * a.n3), g, NT, smem, s);
}

// the persistent column pass at a fixed length: launch it, or (occ) its blocks per SM
template <typename T, int CT, int LF>
static cudaError_t colp_mode(const ColArgs<T>& a, int mode, dim3 g, int nthr, size_t smem, cudaStream_t s, int* occ) {
  constexpr int NT = col_block(ColPlan<LF>::T, 3 * CT, sizeof(T) == 8);
  if (nthr != NT) return cudaErrorNotSupported;
  switch (mode) {
    case COL_Y_FWD: return colp_one<T, CT, COL_Y_FWD, LF, NT>(a, g, smem, s, occ);
    case COL_Y_INV: return colp_one<T, CT, COL_Y_INV, LF, NT>(a, g, smem, s, occ);
    case COL_Z_GREEN: return colp_one<T, CT, COL_Z_GREEN, LF, NT>(a, g, smem, s, occ);
    default: return cudaErrorNotSupported;
  }
}

template <typename T, int CT>
static cudaError_t colp_dispatch(const ColArgs<T>& a, int mode, int L, dim3 g, int nthr, size_t smem, cudaStream_t s,
                                 int* occ) {
  switch (L) {
#define HS_CASE(LEN) case LEN: return colp_mode<T, CT, LEN>(a, mode, g, nthr, smem, s, occ);
    HS_PERSISTENT_LENGTHS(HS_CASE)
#undef HS_CASE
    default: return cudaErrorNotSupported;
  }
}

template <typename T, int MODE, int LF, bool BATCH>
static cudaError_t row_launch(const RowArgs<T>& a, dim3 nb, int nthr, size_t smem, cudaStream_t s) {
  auto k = k_row<T, MODE, LF, BATCH>;
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  return launch_pass(k, a, pass_dependent<T>(a.zstride, (size_t)a.n1 * a.nrows / 3), nb, nthr, smem, s);
}

template <typename T, int MODE, int LF = 0>
static cudaError_t row_one(const RowArgs<T>& a, dim3 nb, int nthr, size_t smem, cudaStream_t s) {
  if (a.zstride != 0) return row_launch<T, MODE, LF, true>(a, nb, nthr, smem, s);
  return row_launch<T, MODE, LF, false>(a, nb, nthr, smem, s);
}

template <typename T, int MODE, int LF = 0, bool BATCH = false>
static cudaError_t row_occ_one(int nthr, size_t smem, int* n) {
  auto k = k_row<T, MODE, LF, BATCH>;
  cudaError_t e = set_smem(k, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, nthr, smem);
}

// compile-time variants for 256-thread blocks at the lengths that have a plan
template <typename T, int MODE>
static cudaError_t row_occ(int n1, int nthr, size_t smem, int* n) {
  if (nthr == 256) {
    switch (n1) {
#define HS_CASE(LEN) case LEN: return row_occ_one<T, MODE, LEN>(nthr, smem, n);
      HS_FIXED_LENGTHS(HS_CASE)
#undef HS_CASE
    }
    if (sizeof(T) == 4 && fft_fixed_length(n1, false)) return launch_row_more(nullptr, MODE, n1, dim3(1), nthr, smem, nullptr, n);
  }
  if (n1 % 5 == 0 || n1 % 7 == 0 || n1 % 11 == 0) return row_blocks_per_sm_ext<T>(MODE, nthr, smem, n);
  return row_occ_one<T, MODE>(nthr, smem, n);
}
template <typename T, int MODE>
static cudaError_t row_dispatch(const RowArgs<T>& a, dim3 nb, int nthr, size_t smem, cudaStream_t s) {
  if (nthr == 256) {
    switch (a.n1) {
#define HS_CASE(LEN) case LEN: return row_one<T, MODE, LEN>(a, nb, nthr, smem, s);
      HS_FIXED_LENGTHS(HS_CASE)
#undef HS_CASE
    }
    if constexpr (sizeof(T) == 4) {
      if (fft_fixed_length(a.n1, false)) return launch_row_more(&a, MODE, a.n1, nb, nthr, smem, s, nullptr);
    }
  }
  if (plan_ext(a.plan)) return launch_row_ext<T>(a, MODE, nb, nthr, smem, s);
  return row_one<T, MODE>(a, nb, nthr, smem, s);
}

template <typename T>
__global__ void k_state_export(const typename cplx_t<T>::type* S, double2* out, size_t nrows, int nh, int P) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nrows * nh) return;
  size_t r = i / nh, k = i - r * nh;
  auto v = S[r * P + k];
  out[i] = make_double2((double)v.x, (double)v.y);
}

template <typename T>
__global__ void k_state_import(const double2* in, typename cplx_t<T>::type* S, size_t nrows, int nh, int P) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nrows * P) return;
  size_t r = i / P, k = i - r * P;
  typename cplx_t<T>::type v;
  if ((int)k < nh) {
    double2 d = in[r * nh + k];
    v.x = (T)d.x;
    v.y = (T)d.y;
  } else {
    v.x = 0;
    v.y = 0;
  }
  S[i] = v;
}

}  // namespace hs

// The fused x pass and the state's import and export.
#define HS_INSTANTIATE(T) \
  namespace hs { \
  template <>                                                                                            \
  cudaError_t launch_march<T>(const MarchArgs<T>& a, bool iso, int ty, int mode, dim3 grid, int nthr, size_t smem, \
                              cudaStream_t s) {                                                          \
    if (a.ids == nullptr || a.mat == nullptr || a.st == nullptr || a.partials == nullptr || a.in == nullptr || \
        a.zstride != 0)                                                                                  \
      return cudaErrorInvalidValue;                                                                      \
    if (mode == MODE_EMIT && a.u64 == nullptr) return cudaErrorInvalidValue;                             \
    if (mode == MODE_FORCE && a.out == nullptr) return cudaErrorInvalidValue;                            \
    if (mode == MODE_FIELDS && (a.eps_out == nullptr || a.sig_out == nullptr)) return cudaErrorInvalidValue; \
    switch (ty) {                                                                                        \
      case 2: return march_ty<T, 2>(a, iso, mode, grid, nthr, smem, s);                                  \
      case 4: return march_ty<T, 4>(a, iso, mode, grid, nthr, smem, s);                                  \
      case 8: return march_ty<T, 8>(a, iso, mode, grid, nthr, smem, s);                                  \
      default: return cudaErrorInvalidValue;                                                             \
    }                                                                                                    \
  }                                                                                                      \
  template <>                                                                                            \
  cudaError_t launch_state_export<T>(const typename cplx_t<T>::type* S, double2* out, int n2, int n3,     \
                                     int nh, int P, cudaStream_t s) {                                    \
    size_t nrows = (size_t)3 * n3 * n2, n = nrows * nh;                                                  \
    k_state_export<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(S, out, nrows, nh, P);                 \
    return cudaGetLastError();                                                                           \
  }                                                                                                      \
  template <>                                                                                            \
  cudaError_t launch_state_import<T>(const double2* in, typename cplx_t<T>::type* S, int n2, int n3,      \
                                     int nh, int P, cudaStream_t s) {                                    \
    size_t nrows = (size_t)3 * n3 * n2, n = nrows * P;                                                   \
    k_state_import<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, S, nrows, nh, P);                  \
    return cudaGetLastError();                                                                           \
  }                                                                                                      \
  }

// Column passes.  CT: the wider column tile (CT / 2 is the default).
#define HS_INSTANTIATE_COLS(T, CT) \
  namespace hs { \
  template <> \
  cudaError_t launch_col<T>(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, cudaStream_t s) { \
    if (a.buf == nullptr || a.tw == nullptr || ((mode == COL_Z_GREEN || mode == COL_Z_INV_STATE) && a.S == nullptr)) \
      return cudaErrorInvalidValue; \
    if (ct == (CT)) return plan_ext(a.plan) ? launch_col_ext<T>(a, mode, ct, grid, nthr, smem, s) \
                                            : col_ct<T, CT>(a, mode, grid, nthr, smem, s); \
    if (ct == (CT) / 2) return col_dispatch<T, (CT) / 2>(a, mode, grid, nthr, smem, s); \
    return cudaErrorInvalidValue; \
  } \
  }

// Persistent column passes (default tile CT).
#define HS_INSTANTIATE_COLP(T, CT) \
  namespace hs { \
  template <> \
  cudaError_t launch_colp<T>(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, cudaStream_t s) { \
    if (a.buf == nullptr || a.tw == nullptr || (mode == COL_Z_GREEN && a.S == nullptr)) return cudaErrorInvalidValue; \
    if (ct != (CT) || plan_ext(a.plan) || a.state_smem) return cudaErrorNotSupported; \
    return colp_dispatch<T, CT>(a, mode, col_length(a, mode), grid, nthr, smem, s, nullptr); \
  } \
  template <> \
  cudaError_t colp_blocks_per_sm<T>(int mode, int L, int ct, int nthr, size_t smem, int* n) { \
    if (ct != (CT)) return cudaErrorNotSupported; \
    ColArgs<T> a; \
    memset(&a, 0, sizeof(a)); \
    return colp_dispatch<T, CT>(a, mode, L, dim3(1), nthr, smem, nullptr, n); \
  } \
  }

// Row passes.
#define HS_INSTANTIATE_ROWS(T) \
  namespace hs { \
  template <>                                                                                            \
  cudaError_t launch_row<T>(const RowArgs<T>& a, int mode, dim3 nb, int nthr, size_t smem, cudaStream_t s) { \
    if (a.tw == nullptr || (mode == ROW_C2R ? (a.spec_in == nullptr || (a.real_out == nullptr && a.acc64 == nullptr)) \
                                            : (a.real_in == nullptr || a.spec_out == nullptr)))         \
      return cudaErrorInvalidValue;                                                                      \
    return mode == ROW_C2R ? row_dispatch<T, ROW_C2R>(a, nb, nthr, smem, s)                             \
                           : row_dispatch<T, ROW_R2C>(a, nb, nthr, smem, s);                            \
  }                                                                                                      \
  template <>                                                                                            \
  cudaError_t row_blocks_per_sm<T>(int mode, int n1, int nthr, size_t smem, int* n) {                     \
    return mode == ROW_C2R ? row_occ<T, ROW_C2R>(n1, nthr, smem, n) : row_occ<T, ROW_R2C>(n1, nthr, smem, n); \
  }                                                                                                      \
  }

// A group of the FP32-only lengths: column passes (cases of launch_col_more's switch) and row passes, whose
// kernels serve single and batched launches.
#define HS_COL_MORE_CASE(LEN)                                                                             \
  case LEN: return col_ct<float, 8, LEN, col_block(ColPlan<LEN>::T, 24, false)>(a, mode, grid, nthr, smem, s);
#define HS_ROW_MORE_CASE(LEN)                                                                             \
  case LEN:                                                                                              \
    if (occ != nullptr) return row_occ_one<float, MODE, LEN, true>(nthr, smem, occ);                      \
    return row_launch<float, MODE, LEN, true>(*a, nb, nthr, smem, s);

// Kernels for plans with a radix-5, 7 or 11 stage, in their own translation unit.
#define HS_INSTANTIATE_EXT(T, CT)                                                                         \
  namespace hs {                                                                                         \
  template <>                                                                                            \
  cudaError_t launch_col_ext<T>(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, \
                                cudaStream_t s) {                                                        \
    if (ct != (CT)) return cudaErrorInvalidValue;                                                        \
    return col_ct<T, CT, -1>(a, mode, grid, nthr, smem, s);                                              \
  }                                                                                                      \
  template <>                                                                                            \
  cudaError_t launch_row_ext<T>(const RowArgs<T>& a, int mode, dim3 nb, int nthr, size_t smem, cudaStream_t s) { \
    return mode == ROW_C2R ? row_one<T, ROW_C2R, -1>(a, nb, nthr, smem, s)                               \
                           : row_one<T, ROW_R2C, -1>(a, nb, nthr, smem, s);                              \
  }                                                                                                      \
  template <>                                                                                            \
  cudaError_t row_blocks_per_sm_ext<T>(int mode, int nthr, size_t smem, int* n) {                        \
    return mode == ROW_C2R ? row_occ_one<T, ROW_C2R, -1>(nthr, smem, n)                                  \
                           : row_occ_one<T, ROW_R2C, -1>(nthr, smem, n);                                 \
  }                                                                                                      \
  }
