// Shared device-side definitions of the tetrahedral-stencil solver.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft.cuh"

namespace hs {

// Device-resident solve status.  Written by the last block of every
// residual-evaluating kernel (see finalize()); read by every other kernel at
// entry so that the work queued after convergence becomes a no-op.
struct DevStatus {
  int done;       // 0 running, 1 converged, 2 max_iter reached, 3 diverged
  int evals;      // residual evaluations so far
  int max_iter;   // stop (done = 2) after this many evaluations
  int hist_cap;   // capacity of the error history
  unsigned int counter;  // block-arrival counter of the last-block reduction
  int retired;    // batched solves: this item is finished and every kernel skips it
  double tol;       // converged when err < tol
  double err;       // error of the last evaluation, Eq. (tolerance)
  double l2;        // L2 norm of the nodal force, Eq. (L2-norm)
  double sig_norm;  // Frobenius norm of <sigma>
  double sig_mean[6];  // <sigma> = 1/2(<sigma^T1> + <sigma^T2>), Voigt order
  double err_min;
  double denom;     // > 0: use this instead of sig_norm (correction solves)
  double nvox;      // N
  // Applied-stress control (Section 2.5, Algorithm 1 step 6): when macro is
  // not null it points at [sigma^a (6, Voigt), S0 (6x6)], S0 mapping a Voigt
  // stress to the tensor strain components of (lambda0)^-1 : sigma, and every
  // evaluation that does not stop moves the macroscopic strain E (tensor
  // components, read by the kernels of the next evaluation) by
  // S0 (sigma^a - <sigma>).
  const double* macro;
  double E[6];
  // > 0: also converged once err <= rel_tol * (err of the first evaluation of this run)
  double rel_tol;
  double err_first;
};

// DONE_TIMEOUT: a bounded device wait (the mbarrier of a tensor copy) gave up; DONE_FAULT: a
// kernel's own check (the alignment a tensor copy needs) failed before the access.  Both stay set.
enum { DONE_RUNNING = 0, DONE_CONVERGED = 1, DONE_MAXITER = 2, DONE_DIVERGED = 3, DONE_TIMEOUT = 4, DONE_FAULT = 5 };

// Programmatic dependents: once every block of a pass has called pass_begin or ended, the next pass's blocks may start;
// pass_wait holds them until this pass has finished and its writes are visible.  Every kernel
// launched as a dependent calls pass_wait before it ends, so that finished means the whole chain before it,
// and until then touches only what no kernel writes: its arguments, shared memory and the twiddle
// tables.  Called early, pass_begin packs the next pass's blocks onto the SMs that are free first: 64^3 FP64
// 277 -> 442 us per evaluation, 256^3 FP32 650 -> 689.  So a pass calls it before its last transform.
__device__ __forceinline__ void pass_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pass_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// FP32 passes of a solve over 2^17 to 2^22 voxels launch as programmatic dependents of the kernel before them:
// their blocks start and fill their twiddle tables while that kernel's last transforms run, and wait for its
// results in pass_wait.  us per evaluation: 64^3 37.2 -> 34.5, 96^3 60.7 -> 58.5, 128^3 101.4 -> 97.5, but
// 44^3 46.1 -> 47.5 (fewer blocks than SMs, some of which then get two), 192^3 328 -> 326 and 256^3 651 -> 655;
// in FP64, whose passes need their blocks spread evenly over the SMs, 64^3 277 -> 326 and 128^3 1749 -> 1894.
// The real-space pass is launched plainly for the same reason, and so are a batch's passes.
template <typename T> __host__ __device__ constexpr bool pass_dependent(size_t zstride, size_t voxels) {
  return sizeof(T) == 4 && zstride == 0 && voxels >= ((size_t)1 << 17) && voxels <= ((size_t)1 << 22);
}

// Batched launches (one launch over many solves of the same grid): item
// blockIdx.z works in the workspace that starts zstride bytes after item
// blockIdx.z - 1's, so every workspace pointer of the launch moves by
// blockIdx.z * zstride.  zstride = 0: a single solve.
template <typename P> __device__ __forceinline__ P* zshift(P* p, size_t off) {
  return p == nullptr ? p : reinterpret_cast<P*>(reinterpret_cast<uintptr_t>(p) + off);
}
constexpr int NRED = 7;  // sum of sigma^T1 + sigma^T2 (6), sum |F|^2 (1)
constexpr int kPartStride = 8;                       // a block's partial sums in memory: NRED values, one spare
constexpr size_t kReduceScratch = 32 * kPartStride * 8;  // shared memory of reduce_and_finalize

// Phase tables.  Isotropic phases: FP32 (lambda, lambda, mu, mu), one 16-byte load of the pairs that
// the two-lane arithmetic takes; FP64 (lambda, mu).  Anisotropic phases: the 21 upper-triangle entries
// of the 6x6 Voigt stiffness, row-major, padded to whole 16-byte loads.
// The stored stiffness is kTabScale times the material's (a power of two; see real.cuh).
template <typename T> constexpr T kTabScale = T(0.0625);
template <typename T> constexpr int kIsoStride = sizeof(T) == 4 ? 4 : 2;
template <typename T> constexpr int kAnisoStride = sizeof(T) == 4 ? 24 : 22;
__device__ __forceinline__ void iso_pairs(const float* tab, int ph, float2& lam, float2& mu) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(tab) + ph);
  lam = make_float2(v.x, v.y);
  mu = make_float2(v.z, v.w);
}
__device__ __forceinline__ void iso_pairs(const double* tab, int ph, double2& lam, double2& mu) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(tab) + ph);
  lam = make_double2(v.x, v.x);
  mu = make_double2(v.y, v.y);
}

// Isotropic phases.
template <typename T> struct MatIso {
  const T* tab;
  __device__ __forceinline__ void stress(int ph, const T* e, T* s) const {
    typename cplx_t<T>::type lp, mp;
    iso_pairs(tab, ph, lp, mp);
    const T lam = lp.x / kTabScale<T>, mu = mp.x / kTabScale<T>;
    const T lt = lam * (e[0] + e[1] + e[2]);
    const T m2 = mu + mu;
    s[0] = lt + m2 * e[0];
    s[1] = lt + m2 * e[1];
    s[2] = lt + m2 * e[2];
    s[3] = mu * e[3];
    s[4] = mu * e[4];
    s[5] = mu * e[5];
  }
};

// General anisotropic phases.  e is the engineering Voigt strain.
template <typename T> struct MatAniso {
  const T* tab;
  __device__ __forceinline__ void stress(int ph, const T* e, T* s) const {
    const T* c = tab + kAnisoStride<T> * ph;
    T C[21];
#pragma unroll
    for (int i = 0; i < 21; ++i) C[i] = __ldg(c + i) / kTabScale<T>;
    // index of (i,j), i <= j, in the packed upper triangle
#define HS_UT(i, j) ((i) * 6 - ((i) * ((i) - 1)) / 2 + ((j) - (i)))
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      T acc = 0;
#pragma unroll
      for (int j = 0; j < 6; ++j) acc += C[i <= j ? HS_UT(i, j) : HS_UT(j, i)] * e[j];
      s[i] = acc;
    }
#undef HS_UT
  }
};

// Evaluation of the stopping test from the sums of one residual evaluation
// (Eqs. L2-norm, tolerance), by one warp: lane v holds sums[v], v < 6 the sum over
// voxels of sigma^T1 + sigma^T2, v = 6 the sum over corners of |F|^2.  Updates the
// status (error, history, done flag, applied-stress strain update) and clears the
// arrival counter.  The status is read in one go, past L1 (other blocks of this
// launch may have recorded a timeout in it).  The divisions and roots run lane by
// lane: each takes some 25 FP64 instructions, 64 cycles apiece whatever the number
// of active lanes (one thread took 10 in a row, 8 us of a 13 us pass at 64^3).
__device__ inline void finalize_eval(DevStatus* st, double* hist, double sum) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int done0 = __ldcg(&st->done), k = __ldcg(&st->evals), max_iter = __ldcg(&st->max_iter),
            hist_cap = __ldcg(&st->hist_cap);
  const double tol = __ldcg(&st->tol), denom = __ldcg(&st->denom), n = __ldcg(&st->nvox),
               rel_tol = __ldcg(&st->rel_tol), err_min0 = __ldcg(&st->err_min), err_first0 = __ldcg(&st->err_first);
  const double* const macro =
      reinterpret_cast<const double*>(__ldcg(reinterpret_cast<const unsigned long long*>(&st->macro)));
  if (lane == 0) st->counter = 0;
  if (done0 == DONE_TIMEOUT || done0 == DONE_FAULT) return;
  const double mean = (lane < 6 ? 0.5 * sum : sum) / n;  // <sigma> (lanes 0-5), mean |F|^2 (lane 6)
  double nrm2 = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double m = __shfl_sync(kAll, mean, i);
    nrm2 += (i < 3 ? 1.0 : 2.0) * m * m;
  }
  const double root = sqrt(lane == 6 ? mean : nrm2);
  const double l2 = __shfl_sync(kAll, root, 6), nrm = __shfl_sync(kAll, root, 0);
  const double den = denom > 0 ? denom : nrm;
  double err;
  if (den > 0) err = l2 / den;
  else err = (l2 == 0) ? 0.0 : __longlong_as_double(0x7ff0000000000000LL);
  if (lane < 6) st->sig_mean[lane] = mean;
  int done = DONE_RUNNING;
  const bool bad = !(err == err) || err > 1e300;
  const double err_min = (k == 0 || err < err_min0) ? err : err_min0;
  const double err_first = k == 0 ? err : err_first0;
  if (bad) done = DONE_DIVERGED;
  else if (err < tol || (rel_tol > 0 && err <= rel_tol * err_first)) done = DONE_CONVERGED;
  else if (err > 1e6 * err_min && k > 10) done = DONE_DIVERGED;
  else if (k + 1 >= max_iter) done = DONE_MAXITER;
  if (lane == 0) {
    st->l2 = l2;
    st->sig_norm = nrm;
    st->err = err;
    if (k < hist_cap) hist[k] = err;
    st->evals = k + 1;
    if (!bad) {
      st->err_min = err_min;
      st->err_first = err_first;
    }
    if (done != DONE_RUNNING) atomicMax(&st->done, done);  // a timeout recorded meanwhile stays
  }
  if (macro != nullptr && done == DONE_RUNNING) {
    // E <- (lambda0)^-1 : {sigma^a + (lambda0 - <lambda>) : E - <lambda : deps> + <lambda : eps0>}
    //    = E + (lambda0)^-1 : (sigma^a - <sigma>)   (the same quantity, regrouped), a component per lane
    const int i = lane < 6 ? lane : 0;
    const double d = macro[i] - mean;
    double acc = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) acc += macro[6 + i * 6 + j] * __shfl_sync(kAll, d, j);
    if (lane < 6) st->E[lane] += acc;
  }
}

// Sums of 8 values per thread over the warp, in a fixed order; lane l returns value l / 4.  9 additions per
// lane instead of 8 x 5: each of the first three exchanges also halves the values a lane keeps.  (FP64
// additions run at 2 lanes per SM and clock, so the plain form cost each block of a pass about 2 us.)
template <typename T> __device__ __forceinline__ T warp_sum8(const T (&acc)[8]) {
  const int lane = threadIdx.x & 31;
  T v[4];
  {
    const bool up = (lane & 16) != 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const T keep = up ? acc[4 + i] : acc[i], send = up ? acc[i] : acc[4 + i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
  }
  {
    const bool up = (lane & 8) != 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const T keep = up ? v[2 + i] : v[i], send = up ? v[i] : v[2 + i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
  }
  const bool up = (lane & 4) != 0;
  const T keep = up ? v[1] : v[0], send = up ? v[0] : v[1];
  T s = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// Sums over the block of the warps' sums (warp_sum8), valid in lanes 0..7 of warp 0 (lane v: value v).
// scratch: kReduceScratch bytes of shared memory.  Every thread of the block must call it.
__device__ inline double block_sum8(double s, double* scratch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (blockDim.x + 31) >> 5;
  if ((lane & 3) == 0) scratch[warp * 8 + (lane >> 2)] = s;
  __syncthreads();
  double t = 0;
  if (warp == 0) {
    for (int w = lane >> 3; w < nw; w += 4) t += scratch[w * 8 + (lane & 7)];
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    t += __shfl_xor_sync(0xffffffffu, t, 8);
  }
  return t;
}

// After every block has written its partials: true in the one block that
// arrives last (all partials of the launch visible to it).
__device__ inline bool last_block_arrived(DevStatus* st, unsigned int nblk) {
  __shared__ bool am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int prev = atomicAdd(&st->counter, 1u);
    am_last = (prev == nblk - 1);
  }
  __syncthreads();
  if (am_last) __threadfence();
  return am_last;
}

// Sum the warps' sums (warp_sum8 of NRED values and a zero) over the block and publish them as its partials.
// scratch: kReduceScratch bytes of shared memory.
__device__ inline void publish_partials(double warp_sum, double* partials, double* scratch) {
  const int bid = blockIdx.y * gridDim.x + blockIdx.x;
  const double s = block_sum8(warp_sum, scratch);
  if (threadIdx.x < 8) partials[(size_t)bid * kPartStride + threadIdx.x] = s;
}

// Sum the partials of nblk blocks in a fixed order and evaluate the stopping
// test, by one block: each thread takes every blockDim-th block's partials,
// four 16-byte loads per block and four blocks in flight.
__device__ inline void finalize_partials(int nblk, const double* partials, DevStatus* st, double* hist,
                                         double* scratch) {
  double a8[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) a8[v] = 0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
    const double2* q = reinterpret_cast<const double2*>(partials + (size_t)b * kPartStride);
    double2 d[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) d[v] = __ldcg(q + v);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      a8[2 * v] += d[v].x;
      if (v < 3) a8[2 * v + 1] += d[v].y;
    }
  }
  const double t = block_sum8(warp_sum8(a8), scratch);
  if (threadIdx.x < 32) finalize_eval(st, hist, t);
}

// Publish this block's partials; the last block to arrive takes the sum and the
// stopping test (passes that no kernel of the same evaluation follows).
__device__ inline void reduce_and_finalize(double warp_sum, double* partials, DevStatus* st, double* hist,
                                           double* scratch) {
  const int nblk = gridDim.x * gridDim.y;
  publish_partials(warp_sum, partials, scratch);
  if (!last_block_arrived(st, (unsigned)nblk)) return;
  finalize_partials(nblk, partials, st, hist, scratch);
}

// ---- mbarriers and tensor (TMA) copies ------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// makes the initialised barriers visible to the async proxy (then a block barrier)
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// Wait for the completion of the barrier phase of the given parity, at most about 2^22 tries
// (each try may suspend the thread for a while); false if the bound ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
  const uint32_t b = smem_u32(bar);
  for (int i = 0; i < (1 << 22); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
// Tiled tensor copy global -> shared of the box at coordinates (c0 .. c4) of a rank-5 tensor map
// (a __grid_constant__ kernel parameter), completing on the mbarrier.  The innermost coordinate
// times the element size must be a multiple of 16 bytes; dst 128-byte aligned.
__device__ __forceinline__ void tma_load_5d(void* dst, const void* tmap, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
      "%6}], [%7];\n" ::"r"(smem_u32(dst)),
      "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}

}  // namespace hs
