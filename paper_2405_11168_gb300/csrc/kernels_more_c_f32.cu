// FP32 column and row passes of lengths 160, 176, 224, 240.
#include "kernels_impl.cuh"

namespace hs {

cudaError_t launch_col_more_c(const ColArgs<float>& a, int mode, int L, dim3 grid, int nthr, size_t smem, cudaStream_t s) {
  switch (L) {
    HS_COL_MORE_CASE(160)
    HS_COL_MORE_CASE(176)
    HS_COL_MORE_CASE(224)
    HS_COL_MORE_CASE(240)
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE>
static cudaError_t row_more(const RowArgs<float>* a, int L, dim3 nb, int nthr, size_t smem, cudaStream_t s, int* occ) {
  switch (L) {
    HS_ROW_MORE_CASE(160)
    HS_ROW_MORE_CASE(176)
    HS_ROW_MORE_CASE(224)
    HS_ROW_MORE_CASE(240)
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t launch_row_more_c(const RowArgs<float>* a, int mode, int L, dim3 nb, int nthr, size_t smem, cudaStream_t s,
                              int* occ) {
  return mode == ROW_C2R ? row_more<ROW_C2R>(a, L, nb, nthr, smem, s, occ) : row_more<ROW_R2C>(a, L, nb, nthr, smem, s, occ);
}

}  // namespace hs
