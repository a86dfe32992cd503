// FP32 fused x pass and state import / export.
#include "kernels_impl.cuh"
HS_INSTANTIATE(float)

namespace hs {

cudaError_t launch_col_more_a(const ColArgs<float>&, int, int, dim3, int, size_t, cudaStream_t);
cudaError_t launch_col_more_b(const ColArgs<float>&, int, int, dim3, int, size_t, cudaStream_t);
cudaError_t launch_col_more_c(const ColArgs<float>&, int, int, dim3, int, size_t, cudaStream_t);
cudaError_t launch_row_more_a(const RowArgs<float>*, int, int, dim3, int, size_t, cudaStream_t, int*);
cudaError_t launch_row_more_b(const RowArgs<float>*, int, int, dim3, int, size_t, cudaStream_t, int*);
cudaError_t launch_row_more_c(const RowArgs<float>*, int, int, dim3, int, size_t, cudaStream_t, int*);

// the FP32-only lengths in three translation units
cudaError_t launch_col_more(const ColArgs<float>& a, int mode, int L, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  return (L <= 80 ? launch_col_more_a : L <= 144 ? launch_col_more_b : launch_col_more_c)(a, mode, L, g, nthr, smem, s);
}
cudaError_t launch_row_more(const RowArgs<float>* a, int mode, int L, dim3 g, int nthr, size_t smem, cudaStream_t s,
                            int* occ) {
  return (L <= 80 ? launch_row_more_a : L <= 144 ? launch_row_more_b : launch_row_more_c)(a, mode, L, g, nthr, smem, s, occ);
}

}  // namespace hs
