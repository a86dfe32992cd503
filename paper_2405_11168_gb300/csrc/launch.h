// Internal launch interface between the C-ABI host code and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "colpass.cuh"
#include "march.cuh"
#include "rowpass.cuh"

namespace hs {

// Entries of the phase tables (layouts in common.cuh): an isotropic phase, or the 21 upper-triangle entries
// of a 6x6 matrix, row-major; rounded to T, then scaled (exactly).
inline void pack_iso(double lam, double mu, double* out) {
  out[0] = lam * kTabScale<double>;
  out[1] = mu * kTabScale<double>;
}
inline void pack_iso(double lam, double mu, float* out) {
  out[0] = out[1] = (float)lam * kTabScale<float>;
  out[2] = out[3] = (float)mu * kTabScale<float>;
}
template <typename T> void pack_upper(const double* C, T* out) {
  for (int i = 0; i < 6; ++i)
    for (int j = i; j < 6; ++j) *out++ = (T)C[i * 6 + j] * kTabScale<T>;
}

// fused x pass (xfuse = 1); mode: MODE_FORCE / MODE_FIELDS / MODE_EMIT
template <typename T>
cudaError_t launch_march(const MarchArgs<T>& a, bool iso, int ty, int mode, dim3 grid, int nthr, size_t smem,
                         cudaStream_t s);

// Compile-time row pitch of the pass on a real displacement: the FP32 force pass with tiles of 4 rows runs
// the next of four; 0: none.
inline int real_pitch_class(bool f64, int ty, int mode, int n1) {
  if (f64 || ty != 4 || mode != MODE_FORCE) return 0;
  return n1 <= 64 ? 64 : n1 <= 128 ? 128 : n1 <= 256 ? 256 : 512;
}
// FP64 tiles of 8 rows of more than 256 columns: two blocks of a cluster take half the columns each
// (N1 a multiple of 16, so that bulk copies take half rows).  The columns and threads of a block.
inline bool real_split(bool f64, int ty, int n1) { return f64 && ty == 8 && n1 > 256; }
inline bool real_rows_fit(bool f64, int ty, int n1) { return !real_split(f64, ty, n1) || n1 % 16 == 0; }
inline int real_halves(bool f64, int ty, int n1) { return real_split(f64, ty, n1) ? 2 : 1; }
inline int real_threads(bool f64, int ty, int n1) { return (n1 / real_halves(f64, ty, n1) + 31) / 32 * 32; }
// Its row pitch in shared memory.
inline int real_pitch(bool f64, int ty, int mode, int n1) {
  const int c = real_pitch_class(f64, ty, mode, n1);
  return c > 0 ? c : real_split(f64, ty, n1) ? n1 / 2 + 8 : (n1 + 7) & ~7;
}

// The pass on a real displacement field (k_real): mode MODE_FORCE / MODE_FIELDS / MODE_FORCE_FIELDS (FP64
// only); grid: (N2 / ty * real_halves(), z chunks, items), real_threads() threads; a.xp as real_pitch() gives it.  occ: not null: the resident blocks per SM instead of a launch.
template <typename T, bool ISO>
cudaError_t launch_real_law(const MarchArgs<T>& a, int ty, int mode, dim3 grid, int nthr, size_t smem, cudaStream_t s,
                            int* occ);
template <> cudaError_t launch_real_law<float, true>(const MarchArgs<float>&, int, int, dim3, int, size_t, cudaStream_t, int*);
template <> cudaError_t launch_real_law<float, false>(const MarchArgs<float>&, int, int, dim3, int, size_t, cudaStream_t, int*);
template <> cudaError_t launch_real_law<double, true>(const MarchArgs<double>&, int, int, dim3, int, size_t, cudaStream_t, int*);
template <> cudaError_t launch_real_law<double, false>(const MarchArgs<double>&, int, int, dim3, int, size_t, cudaStream_t, int*);
template <typename T>
cudaError_t launch_real(const MarchArgs<T>& a, bool iso, int ty, int mode, dim3 grid, int nthr, size_t smem,
                        cudaStream_t s, int* occ = nullptr) {
  return iso ? launch_real_law<T, true>(a, ty, mode, grid, nthr, smem, s, occ)
             : launch_real_law<T, false>(a, ty, mode, grid, nthr, smem, s, occ);
}

template <typename T>
cudaError_t launch_col(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, cudaStream_t s);

// persistent double-buffered column pass (COL_Y_FWD, COL_Y_INV, COL_Z_GREEN) for the compile-time
// lengths 128, 192, 256, 384, 512 with the default tile and block size: grid.x persistent blocks,
// grid.z items; cudaErrorNotSupported when no such variant exists
template <typename T>
cudaError_t launch_colp(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, cudaStream_t s);
template <typename T>
cudaError_t colp_blocks_per_sm(int mode, int L, int ct, int nthr, size_t smem, int* n);

// mode: ROW_C2R / ROW_R2C; grid.x persistent blocks per item, grid.z items (batched launches)
template <typename T>
cudaError_t launch_row(const RowArgs<T>& a, int mode, dim3 grid, int nthr, size_t smem, cudaStream_t s);

// column and row passes of the FP32-only compile-time lengths; a null: *occ = resident blocks per SM
cudaError_t launch_col_more(const ColArgs<float>& a, int mode, int L, dim3 grid, int nthr, size_t smem, cudaStream_t s);
cudaError_t launch_row_more(const RowArgs<float>* a, int mode, int L, dim3 grid, int nthr, size_t smem, cudaStream_t s,
                            int* occ);

// the same passes for plans with a radix-5, 7 or 11 stage (default column tile only)
template <typename T>
cudaError_t launch_col_ext(const ColArgs<T>& a, int mode, int ct, dim3 grid, int nthr, size_t smem, cudaStream_t s);
template <typename T>
cudaError_t launch_row_ext(const RowArgs<T>& a, int mode, dim3 grid, int nthr, size_t smem, cudaStream_t s);
template <typename T>
cudaError_t row_blocks_per_sm_ext(int mode, int nthr, size_t smem, int* n);

// resident blocks per SM of the row pass (persistent grid sizing)
template <typename T>
cudaError_t row_blocks_per_sm(int mode, int n1, int nthr, size_t smem, int* n);

// u8 phase ids -> u16
cudaError_t launch_ids_u8_to_u16(const uint8_t* in, uint16_t* out, size_t n, cudaStream_t s);
// widen a float array to double
cudaError_t launch_f32_to_f64(const float* in, double* out, size_t n, cudaStream_t s);
// largest id into *out (int, must start at 0)
cudaError_t launch_max_id(const uint16_t* ids, size_t n, int* out, cudaStream_t s);
// padded T-complex state <-> packed complex128 [3][n3][n2][nh]
template <typename T>
cudaError_t launch_state_export(const typename cplx_t<T>::type* S, double2* out, int n2, int n3, int nh, int P,
                                cudaStream_t s);
template <typename T>
cudaError_t launch_state_import(const double2* in, typename cplx_t<T>::type* S, int n2, int n3, int nh, int P,
                                cudaStream_t s);

}  // namespace hs
