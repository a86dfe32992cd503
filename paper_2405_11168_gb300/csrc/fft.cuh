// Batched mixed-radix (2/3/4/8/16, and 5/7/11) complex FFTs on sequences held in shared memory.
//
// Self-sorting Stockham formulation, one radix-R butterfly per (thread, step):
// stage s with radix R and Ns = R_1...R_{s-1} reads x[b + m L/R], multiplies by
// the twiddle w_{Ns R}^{(b mod Ns) m}, takes a length-R DFT and writes
// y[(b div Ns) Ns R + (b mod Ns) + m Ns].  After the last stage the result is in
// natural order.  Every stage is done in place: a thread loads all of its
// butterflies' inputs into registers, the block synchronises, then it writes.
//
// Run-time plans: ceil(L/kE) threads per sequence with kE = 8 elements per thread,
// so a thread never holds more than ceil(kE/R) butterflies of one stage; radices
// are 8, 4, 3 and 2, and 5, 7 and 11 in kernels of their own.  Compile-time plans
// (below) choose their threads and take radices up to 16.  Length-5, 7 and 11 DFTs fold the mirrored
// inputs and use constant coefficients (DftPrime).  Sequence s, element e lives at
// buf[s*ss + e*es].  Forward = exp(-2 pi i nk/L), inverse = exp(+...), both
// unnormalised.  Twiddles come from a per-axis table w_L^j = exp(-2 pi i j/L),
// j < L, computed on the host.
#pragma once
#include <cuda_runtime.h>

namespace hs {

template <typename T> struct cplx_t;
template <> struct cplx_t<float> { using type = float2; };
template <> struct cplx_t<double> { using type = double2; };

template <typename C> __device__ __forceinline__ C cmk(decltype(C::x) a, decltype(C::x) b) { C r; r.x = a; r.y = b; return r; }
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return cmk<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return cmk<C>(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return cmk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cscale(C a, decltype(C::x) s) { return cmk<C>(a.x * s, a.y * s); }
template <typename C> __device__ __forceinline__ C cconj(C a) { return cmk<C>(a.x, -a.y); }
// multiply by -i (forward quarter turn) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C rot90(C a) {
  return INV ? cmk<C>(-a.y, a.x) : cmk<C>(a.y, -a.x);
}

// cos and sin of 2 pi J / 16 (exact constants of the regular 16-gon)
#define HS_FFT_C1 0.92387953251128675613
#define HS_FFT_S1 0.38268343236508977173
#define HS_FFT_H 0.70710678118654752440
__host__ __device__ constexpr double cos16c(int j) {
  return ((j & 15) == 0) ? 1.0 : ((j & 15) == 1) ? HS_FFT_C1 : ((j & 15) == 2) ? HS_FFT_H : ((j & 15) == 3) ? HS_FFT_S1
       : ((j & 15) == 4) ? 0.0 : ((j & 15) == 5) ? -HS_FFT_S1 : ((j & 15) == 6) ? -HS_FFT_H : ((j & 15) == 7) ? -HS_FFT_C1
       : ((j & 15) == 8) ? -1.0 : ((j & 15) == 9) ? -HS_FFT_C1 : ((j & 15) == 10) ? -HS_FFT_H : ((j & 15) == 11) ? -HS_FFT_S1
       : ((j & 15) == 12) ? 0.0 : ((j & 15) == 13) ? HS_FFT_S1 : ((j & 15) == 14) ? HS_FFT_H : HS_FFT_C1;
}
// sin(t) = cos(t + 3 pi / 2)
__host__ __device__ constexpr double sin16c(int j) { return cos16c(j + 12); }
// w16^J for the requested direction (forward: exp(-2 pi i J/16))
template <int J, bool INV, typename C> __device__ __forceinline__ C w16() {
  using R = decltype(C::x);
  constexpr double c = cos16c(J), sn = sin16c(J);
  return cmk<C>((R)c, INV ? (R)sn : (R)-sn);
}

template <int R, bool INV, typename C> struct Dft;

template <bool INV, typename C> struct Dft<2, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    C a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <bool INV, typename C> struct Dft<3, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    using R = decltype(C::x);
    const R h = (R)0.86602540378443864676;  // sqrt(3)/2
    C s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    C x0 = v[0];
    C m = cmk<C>(x0.x - (R)0.5 * s.x, x0.y - (R)0.5 * s.y);
    // forward: X1 = m - i h d, X2 = m + i h d
    C ihd = cmk<C>(-h * d.y, h * d.x);  // i h d
    v[0] = cadd(x0, s);
    if (INV) {
      v[1] = cadd(m, ihd);
      v[2] = csub(m, ihd);
    } else {
      v[1] = csub(m, ihd);
      v[2] = cadd(m, ihd);
    }
  }
};

template <bool INV, typename C> struct Dft<4, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    C t2 = cadd(v[1], v[3]), t3 = rot90<INV>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  }
};

// composite DFT of length A*B: n = B n1 + n2, k = k1 + A k2
template <int A, int B, bool INV, typename C, int N2 = 1, int K1 = 1>
__device__ __forceinline__ void twiddle_all(C (&y)[B][A]) {
  if constexpr (N2 < B) {
    if constexpr (K1 < A) {
      y[N2][K1] = cmul(y[N2][K1], w16<(16 / (A * B)) * N2 * K1, INV, C>());
      twiddle_all<A, B, INV, C, N2, K1 + 1>(y);
    } else {
      twiddle_all<A, B, INV, C, N2 + 1, 1>(y);
    }
  }
}

template <int A, int B, bool INV, typename C> __device__ __forceinline__ void dft_composite(C* v) {
  C y[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) y[n2][n1] = v[B * n1 + n2];
    Dft<A, INV, C>::run(y[n2]);
  }
  twiddle_all<A, B, INV, C>(y);
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C z[B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) z[n2] = y[n2][k1];
    Dft<B, INV, C>::run(z);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = z[k2];
  }
}

// DFT of length A*B, A and B coprime, without twiddles (prime factor map): n = B n1 + A n2,
// k = k1 (mod A), k = k2 (mod B).  U = B^-1 mod A, V = A^-1 mod B.
template <int A, int B, int U, int V, bool INV, typename C> __device__ __forceinline__ void dft_coprime(C* v) {
  static_assert((B * U) % A == 1 % A && (A * V) % B == 1 % B, "inverse residues");
  constexpr int N = A * B;
  C y[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) y[n2][n1] = v[(B * n1 + A * n2) % N];
    Dft<A, INV, C>::run(y[n2]);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C z[B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) z[n2] = y[n2][k1];
    Dft<B, INV, C>::run(z);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[(B * U * k1 + A * V * k2) % N] = z[k2];
  }
}
template <bool INV, typename C> struct Dft<6, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_coprime<2, 3, 1, 2, INV>(v); }
};
template <bool INV, typename C> struct Dft<12, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_coprime<3, 4, 1, 3, INV>(v); }
};

template <bool INV, typename C> struct Dft<10, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_coprime<2, 5, 1, 3, INV>(v); }
};
template <bool INV, typename C> struct Dft<14, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_coprime<2, 7, 1, 4, INV>(v); }
};

// cos and sin of 2 pi j / P, 1 <= j <= (P - 1) / 2, for the odd prime radices
template <int P> __host__ __device__ constexpr double prime_cos(int j) {
  if (P == 5) return j == 1 ? 0.30901699437494745 : -0.8090169943749473;
  if (P == 7) return j == 1 ? 0.6234898018587336 : j == 2 ? -0.22252093395631434 : -0.900968867902419;
  return j == 1 ? 0.8412535328311812 : j == 2 ? 0.41541501300188644 : j == 3 ? -0.142314838273285
       : j == 4 ? -0.654860733945285 : -0.9594929736144974;
}
template <int P> __host__ __device__ constexpr double prime_sin(int j) {
  if (P == 5) return j == 1 ? 0.9510565162951535 : 0.5877852522924732;
  if (P == 7) return j == 1 ? 0.7818314824680298 : j == 2 ? 0.9749279121818236 : 0.43388373911755823;
  return j == 1 ? 0.5406408174555976 : j == 2 ? 0.9096319953545183 : j == 3 ? 0.9898214418809328
       : j == 4 ? 0.7557495743542583 : 0.28173255684142967;
}
// The same at any multiple, folded to the first half turn.
template <int P> __host__ __device__ constexpr double prime_cos_at(int jk) {
  const int r = jk % P;
  return r == 0 ? 1.0 : prime_cos<P>(r <= P / 2 ? r : P - r);
}
template <int P> __host__ __device__ constexpr double prime_sin_at(int jk) {
  const int r = jk % P;
  return r == 0 ? 0.0 : r <= P / 2 ? prime_sin<P>(r) : -prime_sin<P>(P - r);
}
// Odd prime length: sums and differences of the mirrored inputs, then (P - 1) / 2 real combinations for
// each mirrored pair of outputs, with constant coefficients: (P - 1)^2 multiplications (of reals) where
// the plain sum takes 4 (P - 1)^2 and reads its coefficients from memory.
template <int P, bool INV, typename C> struct DftPrime {
  static __device__ __forceinline__ void run(C* v) {
    using R = decltype(C::x);
    constexpr int H = P / 2;
    C s[H], d[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      s[j] = cadd(v[j + 1], v[P - 1 - j]);
      d[j] = csub(v[j + 1], v[P - 1 - j]);
    }
    const C x0 = v[0];
    C sum = x0;
#pragma unroll
    for (int j = 0; j < H; ++j) sum = cadd(sum, s[j]);
    v[0] = sum;
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      C a = x0, b = cmk<C>(0, 0);
#pragma unroll
      for (int j = 1; j <= H; ++j) {
        const R c = (R)prime_cos_at<P>(j * k), w = (R)prime_sin_at<P>(j * k);
        a = cmk<C>(a.x + c * s[j - 1].x, a.y + c * s[j - 1].y);
        b = cmk<C>(b.x + w * d[j - 1].x, b.y + w * d[j - 1].y);
      }
      const C ib = rot90<INV>(b);  // forward: -i b, inverse: i b
      v[k] = cadd(a, ib);
      v[P - k] = csub(a, ib);
    }
  }
};
template <bool INV, typename C> struct Dft<5, INV, C> : DftPrime<5, INV, C> {};
template <bool INV, typename C> struct Dft<7, INV, C> : DftPrime<7, INV, C> {};
template <bool INV, typename C> struct Dft<11, INV, C> : DftPrime<11, INV, C> {};

template <bool INV, typename C> struct Dft<8, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_composite<2, 4, INV>(v); }
};
template <bool INV, typename C> struct Dft<16, INV, C> {
  static __device__ __forceinline__ void run(C* v) { dft_composite<4, 4, INV>(v); }
};

// Two-float reals (h + l unevaluated, |l| below an ulp of h) for the butterflies of inverse FP32
// transforms whose compile-time plan has a radix-11 stage.  A value there is rounded some nine times at
// full size, and the strain is a difference of the transformed displacement, so that noise is what the FP32
// iteration settles at (44^3: 1.25e-7 of the displacement per evaluation, 5e-6 of the stress in the
// stiff phase).  With the inside of a butterfly in two floats a stage rounds once: 6e-8.
struct df {
  float h, l;
  __device__ __forceinline__ df() {}
  __device__ __forceinline__ constexpr df(double c) : h((float)c), l((float)(c - (double)(float)c)) {}
  __device__ __forceinline__ constexpr df(float h_, float l_) : h(h_), l(l_) {}
};
__device__ __forceinline__ df operator+(df a, df b) {  // the sum of the high parts exactly (Knuth)
  const float s = __fadd_rn(a.h, b.h), z = __fadd_rn(s, -a.h);
  const float e = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -z)), __fadd_rn(b.h, -z));
  return df(s, __fadd_rn(__fadd_rn(a.l, b.l), e));
}
__device__ __forceinline__ df operator-(df a) { return df(-a.h, -a.l); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  return df(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p))));
}
struct cdf {
  df x, y;
};
__device__ __forceinline__ cdf widen(float2 a) {
  cdf r;
  r.x = df(a.x, 0.f);
  r.y = df(a.y, 0.f);
  return r;
}
__device__ __forceinline__ float2 narrow(cdf a) { return make_float2(a.x.h + a.x.l, a.y.h + a.y.l); }

// 16-byte asynchronous global -> shared copies (cp.async, bypassing L1).
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Bulk shared -> global copies (cp.async.bulk, bulk-group completion).  Both
// addresses 16-byte aligned, size a multiple of 16.  The writes that filled
// the shared source must be made visible to the async proxy first
// (fence_async_smem() by every writing thread, then a barrier).
__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, unsigned bytes) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(ssrc));
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(gdst), "r"(s), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// the shared sources of all committed bulk copies may be overwritten
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
// all committed bulk copies are complete
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

constexpr int kMaxStages = 8;
// Radix of each stage packed 4 bits per stage (stage 0 in the low bits), so
// the plan is three plain integers and never needs indexed storage.
struct FftPlan {
  int L;       // sequence length
  int nstage;  // number of radix stages (<= kMaxStages)
  int packed;  // radix of stage s = (packed >> 4 s) & 15, product = L
};

// One Stockham stage over the sequences handled by this thread.
constexpr int kE = 8;

template <int R, bool INV, typename C>
__device__ __forceinline__ void stockham_stage(C* buf, int ss, int es, int ps, int s, int t, int T, bool active,
                                               int L, int Ns, int nsh, const C* __restrict__ tw, bool wsync) {
  // element e of sequence s lives at buf[s*ss + e*es + (ps >= 0 ? e >> ps : 0)]
  // nsh >= 0: Ns = 2^nsh (shift/mask index math), else generic division
  constexpr int KB = (kE + R - 1) / R;
  C v[KB][R];
  const int nb = L / R;
  const int step = L / (Ns * R);
  C* sb = buf + s * ss;
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = t + k * T;
    if (active && b < nb) {
#pragma unroll
      for (int m = 0; m < R; ++m) {
        const int e = b + m * nb;
        v[k][m] = sb[e * es + (ps >= 0 ? (e >> ps) : 0)];
      }
    }
  }
  if (wsync) __syncwarp(); else __syncthreads();
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = t + k * T;
    if (active && b < nb) {
      const int kk = (nsh >= 0) ? (b & (Ns - 1)) : (b % Ns);
      const int pq = (nsh >= 0) ? (b >> nsh) : (b / Ns);
      if (Ns > 1) {
#pragma unroll
        for (int m = 1; m < R; ++m) {
          C w = __ldg(tw + kk * m * step);
          if (INV) w.y = -w.y;
          v[k][m] = cmul(v[k][m], w);
        }
      }
      const int base = pq * Ns * R + kk;
      Dft<R, INV, C>::run(v[k]);
#pragma unroll
      for (int m = 0; m < R; ++m) {
        const int e = base + m * Ns;
        sb[e * es + (ps >= 0 ? (e >> ps) : 0)] = v[k][m];
      }
    }
  }
  if (wsync) __syncwarp(); else __syncthreads();
}

// FFT of nseq sequences in place.  All threads of the block must call this.
// T = ceil(L/kE) threads per sequence, G = blockDim / T sequences per group.
// COLMAP = false: thread i works on sequence g0 + i / T (lanes walk along one
// sequence: for sequences stored as rows, element stride es = 1, padded with
// ps = 3, i.e. one spare slot per 8 elements).  COLMAP = true: thread i works
// on sequence g0 + i % G (lanes walk across sequences: for column tiles whose
// sequences are adjacent in memory, ss = 1).  Either way a warp's shared-memory
// accesses stay (nearly) free of bank conflicts.
// EXT: also radices 5, 7, 11 (their stages keep more values live, so only the
// kernels instantiated for such lengths carry them).
template <bool INV, bool COLMAP, bool EXT = false, typename C>
__device__ __forceinline__ void fft_smem(C* buf, int ss, int es, int ps, int nseq, int L, int nstage, int packed,
                                         const C* __restrict__ tw, int tid, int nthreads) {
  const int T = (L + kE - 1) / kE;
  const int G = nthreads / T;
  for (int g0 = 0; g0 < nseq; g0 += G) {
    const int sl = COLMAP ? (tid % G) : (tid / T);
    const int t = COLMAP ? (tid / G) : (tid % T);
    const int s = g0 + sl;
    const bool active = (COLMAP ? (t < T) : (sl < G)) && s < nseq;
    // row mapping with T dividing 32: every sequence lives inside one warp,
    // so a warp barrier orders its stages (the caller syncs the block after)
    const bool wsync = !COLMAP && T <= 32 && (32 % T) == 0 && (nthreads % 32) == 0;
    int Ns = 1, nsh = 0;
#pragma unroll 1
    for (int st = 0; st < nstage; ++st) {
      const int R = (packed >> (4 * st)) & 15;
      if (R == 8) stockham_stage<8, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else if (R == 4) stockham_stage<4, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else if (R == 3) stockham_stage<3, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else if (EXT && R == 5) stockham_stage<EXT ? 5 : 2, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else if (EXT && R == 7) stockham_stage<EXT ? 7 : 2, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else if (EXT && R == 11) stockham_stage<EXT ? 11 : 2, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      else stockham_stage<2, INV>(buf, ss, es, ps, s, t, T, active, L, Ns, nsh, tw, wsync);
      Ns *= R;
      nsh = (nsh >= 0 && (R & (R - 1)) == 0) ? nsh + (R == 8 ? 3 : R == 4 ? 2 : 1) : -1;
    }
  }
}

// padded index of element e in a row sequence (one spare slot per 8 elements)
__host__ __device__ __forceinline__ int rpad(int e) { return e + (e >> 3); }
__host__ __device__ __forceinline__ int rpitch(int n) { return n + (n >> 3) + 1; }

#define HS_FFT_ROWS(INV, buf, pitch, nseq, plan, tw, tid, nthr)                                       \
  ::hs::fft_smem<INV, false>(buf, pitch, 1, 3, nseq, (plan).L, (plan).nstage, (plan).packed, tw, tid, nthr)
// a plan with a radix-5, 7 or 11 stage
__host__ __device__ inline bool plan_ext(const FftPlan& p) {
  for (int st = 0; st < p.nstage; ++st) {
    const int R = (p.packed >> (4 * st)) & 15;
    if (R == 5 || R == 7 || R == 11) return true;
  }
  return false;
}

#define HS_FFT_COLS(INV, buf, W, nseq, plan, tw, tid, nthr) \
  ::hs::fft_smem<INV, true>(buf, 1, W, -1, nseq, (plan).L, (plan).nstage, (plan).packed, tw, tid, nthr)


// ---------------------------------------------------------------------------
// Compile-time plans: every stride, stage count and radix is a constant, so
// the per-element index arithmetic folds away.  A plan is its radices and the
// number of threads T that share a sequence; T divides L / r for every radix r
// where it can, so that no thread idles in any stage.  A thread holds about
// L / T values.
// Few stages of large radices: a stage costs a load and a store of every value
// through shared memory and two barriers.  Measured per pass (us, FP32, cubes): columns 128 as 8 x 16 15.5 y
// and 27.5 z (8 x 4 x 4: 18.8, 38.7), 192 as 8 x 4 x 6 with 8 threads 35, 91 (4 x 4 x 12 with 16: 47, 110;
// run-time plan 80, 166), 96 as 8 x 12 8.1, 11.0 (4 x 4 x 6: 8.1, 13.0; run-time plan 13, 21), 256 as 8 x 8 x 4
// 78, 188 (16 x 16: 78, 217); rows 256 as 16 x 16 81 and 73 (8 x 8 x 4: 87, 78), 192 as 4 x 4 x 12 48
// (8 x 4 x 6: 67; run-time plan 84), 96 as 4 x 4 x 6 10.5 (8 x 12: 11.8), 128 in FP64 as 8 x 4 x 4 158 (8 x 16: 179).
// ---------------------------------------------------------------------------
// Further FP32 lengths, most with a factor 5, 7 or 11: as the run-time plan, whose index arithmetic, predicates and
// radix switch cost three times the butterflies, a y pass of 112 took 38 us, a z pass of 88 58 and an x pass of
// 160 37 (160 x 112 x 88).  The list is a choice and no measured line: lengths up to 240 with a plan of two (240:
// three) stages of radices up to 16, most of them multiples of 8, at about 1.5 MB of library each.  168, 200,
// 216, 264, 280, 288, 320 and the lengths between have none and run the run-time plan.
template <int LEN, int THREADS, int NST, int R0, int R1, int R2 = 1, int R3 = 1> struct FixedPlan {
  static constexpr int L = LEN, n = NST, T = THREADS;
  __host__ __device__ static constexpr int r(int i) { return i == 0 ? R0 : i == 1 ? R1 : i == 2 ? R2 : R3; }
  static_assert(R0 * R1 * R2 * R3 == L, "radices");
  static constexpr bool two_float = R0 == 11 || R1 == 11 || R2 == 11;  // see df
};
template <int L> struct ColPlan;
template <> struct ColPlan<32> : FixedPlan<32, 4, 2, 4, 8> {};
template <> struct ColPlan<48> : FixedPlan<48, 4, 2, 4, 12> {};
template <> struct ColPlan<64> : FixedPlan<64, 8, 2, 8, 8> {};
template <> struct ColPlan<96> : FixedPlan<96, 4, 2, 8, 12> {};
template <> struct ColPlan<128> : FixedPlan<128, 8, 2, 8, 16> {};
template <> struct ColPlan<192> : FixedPlan<192, 8, 3, 8, 4, 6> {};
template <> struct ColPlan<256> : FixedPlan<256, 32, 3, 8, 8, 4> {};
template <> struct ColPlan<384> : FixedPlan<384, 32, 4, 4, 4, 4, 6> {};
template <> struct ColPlan<512> : FixedPlan<512, 64, 3, 8, 8, 8> {};
template <> struct ColPlan<40> : FixedPlan<40, 8, 2, 8, 5> {};
template <> struct ColPlan<44> : FixedPlan<44, 4, 2, 4, 11> {};
template <> struct ColPlan<56> : FixedPlan<56, 8, 2, 8, 7> {};
template <> struct ColPlan<72> : FixedPlan<72, 6, 2, 12, 6> {};
template <> struct ColPlan<80> : FixedPlan<80, 8, 2, 8, 10> {};
template <> struct ColPlan<88> : FixedPlan<88, 8, 2, 8, 11> {};
template <> struct ColPlan<112> : FixedPlan<112, 8, 2, 8, 14> {};
template <> struct ColPlan<120> : FixedPlan<120, 12, 2, 12, 10> {};
template <> struct ColPlan<144> : FixedPlan<144, 12, 2, 12, 12> {};
template <> struct ColPlan<160> : FixedPlan<160, 10, 2, 16, 10> {};
template <> struct ColPlan<176> : FixedPlan<176, 16, 2, 16, 11> {};
template <> struct ColPlan<224> : FixedPlan<224, 16, 2, 16, 14> {};
template <> struct ColPlan<240> : FixedPlan<240, 24, 3, 4, 6, 10> {};
// rows: T a power of two that divides L
template <int L> struct RowPlan : ColPlan<L> {};
template <> struct RowPlan<72> : FixedPlan<72, 8, 2, 12, 6> {};
template <> struct RowPlan<120> : FixedPlan<120, 8, 2, 12, 10> {};
template <> struct RowPlan<144> : FixedPlan<144, 16, 2, 12, 12> {};
template <> struct RowPlan<160> : FixedPlan<160, 16, 2, 16, 10> {};
template <> struct RowPlan<240> : FixedPlan<240, 16, 3, 4, 6, 10> {};
template <> struct RowPlan<96> : FixedPlan<96, 8, 3, 4, 4, 6> {};
template <> struct RowPlan<128> : FixedPlan<128, 16, 3, 8, 4, 4> {};
template <> struct RowPlan<192> : FixedPlan<192, 16, 3, 4, 4, 12> {};
template <> struct RowPlan<256> : FixedPlan<256, 16, 2, 16, 16> {};
#define HS_FIXED_LENGTHS(F) F(32) F(48) F(64) F(96) F(128) F(192) F(256) F(384) F(512)
// FP32 only (FP64 runs their run-time plans: its passes wait for the FP64 pipe, not for the index arithmetic)
#define HS_FIXED_LENGTHS_F32(F) \
  F(40) F(44) F(56) F(72) F(80) F(88) F(112) F(120) F(144) F(160) F(176) F(224) F(240)

// lengths whose column passes also run persistent
#define HS_PERSISTENT_LENGTHS(F) F(128) F(192) F(256) F(384) F(512)

// threads per sequence: the plan's, or one per kE values for the run-time plans
template <template <int> class PLAN> __host__ __device__ inline int fft_threads(int L, bool f64) {
  switch (L) {
#define HS_CASE(LEN) case LEN: return PLAN<LEN>::T;
    HS_FIXED_LENGTHS(HS_CASE)
#undef HS_CASE
#define HS_CASE(LEN) case LEN: if (!f64) return PLAN<LEN>::T; break;
    HS_FIXED_LENGTHS_F32(HS_CASE)
#undef HS_CASE
  }
  return (L + kE - 1) / kE;
}
__host__ __device__ inline bool fft_fixed_length(int L, bool f64) {
  switch (L) {
#define HS_CASE(LEN) case LEN:
    HS_FIXED_LENGTHS(HS_CASE) return true;
    HS_FIXED_LENGTHS_F32(HS_CASE) return !f64;
#undef HS_CASE
    default: return false;
  }
}

__host__ __device__ constexpr int ilog2_c(int v) { return v <= 1 ? 0 : 1 + ilog2_c(v >> 1); }

// values a thread of the plan holds; above 8 the passes ask for fewer resident threads, so that the
// values, a butterfly's temporaries and its twiddles stay in registers
template <class PL> __host__ __device__ constexpr bool fft_wide() { return PL::L > 8 * PL::T; }
// more than 16 values, radix 12, or a long plan with radix 10 to 14 (us y, z with the tighter bound and its
// spills -> this one: 176 40, 166 -> 36, 155; 224 80, 160 -> 63, 147; but 112 12.3, 22 -> 12.6, 26 and
// the z pass of 88 41 -> 47, where the resident threads count for more)
template <class PL> __host__ __device__ constexpr bool fft_very_wide() {
  for (int i = 0; i < 4; ++i)
    if (PL::r(i) == 12 || (PL::L > 160 && PL::r(i) >= 10 && PL::r(i) <= 14)) return true;
  return PL::L > 16 * PL::T;
}

// Block of a column pass over tiles of W sequences: the most sequences at a time that divide W (no thread
// idles in any round) and stay within 256 (FP32) or 192 (FP64) threads; 512 threads for 64 per sequence (FP32 512),
// whose tiles leave room for two blocks per SM only: 512^3 y 826 -> 594 us, z 2295 -> 1868.
__host__ __device__ constexpr int col_block(int T, int W, bool f64) {
  const int limit = f64 ? 192 : T >= 64 ? 512 : 256;
  int g = W;
  while (g > 1 && (W % g != 0 || g * T > limit)) --g;
  return (g * T + 31) / 32 * 32;
}

// Position of element e inside a row (sequence with unit element stride) and the spacing of rows in shared
// memory, chosen so that the 64-bit accesses of a half-warp fall on different banks in every stage:
//  * 32, 64, 128, 512: the XOR swizzle e ^ (((e >> 2) ^ (e >> 3)) & 15), rows of 32 and 64 spaced 36 and 72
//    apart; 256: e ^ ((e >> 4) & 15);
//  * other lengths: one spare slot per T elements (e + e / T, T a power of two), rows spaced by T (mod 16).
template <int L> struct RowPos {
  static constexpr bool pow2 = (L & (L - 1)) == 0;
  static constexpr int T = RowPlan<L>::T;
  static_assert((T & (T - 1)) == 0 && L % T == 0, "row positions");
  static constexpr int padded = L + L / T;
  static constexpr int pitch = L == 32 ? 36 : L == 64 ? 72 : pow2 ? L
                               : padded + (T >= 16 ? 0 : ((T - padded) % 16 + 16) % 16);
  __host__ __device__ static constexpr int at(int e) {
    return L == 256 ? e ^ ((e >> 4) & 15)
         : pow2 ? e ^ (((e >> 2) ^ (e >> 3)) & 15) : e + (e >> ilog2_c(T));
  }
};
__host__ __device__ inline int row_pitch(int L, bool f64) {
  switch (L) {
#define HS_CASE(LEN) case LEN: return RowPos<LEN>::pitch;
    HS_FIXED_LENGTHS(HS_CASE)
#undef HS_CASE
#define HS_CASE(LEN) case LEN: if (!f64) return RowPos<LEN>::pitch; break;
    HS_FIXED_LENGTHS_F32(HS_CASE)
#undef HS_CASE
  }
  return rpitch(L);
}
// The swizzles are linear over XOR (shifts, XOR and masks are), and an index that is a sum of parts with
// disjoint bits is their XOR, so at(a + b) = at(a) ^ at(b) for such parts; the padded positions are
// additive when the second part is a multiple of T and the first below T.  Either way a thread finds its
// own part once per stage and each element adds a constant.
template <int L> __device__ __forceinline__ int row_join(int a, int c) {
  return RowPos<L>::pow2 ? (a ^ c) : (a + c);
}

// b = pq NS + kk (kk < NS) -> pq NS R + kk
template <int NS, int R> __device__ __forceinline__ int stockham_out(int b) {
  return (b / NS) * (NS * R) + b % NS;
}

// Twiddle table of a fixed plan in shared memory, laid out per stage: stage s (NS_s = r_0 ... r_{s-1}
// > 1) needs w_L^{kk m step_s} for m = 1 .. R_s - 1 and kk < NS_s, kept at entry
// NS_s - r_0 + (m - 1) NS_s + kk.  The lanes of a warp hold consecutive kk, so they read consecutive
// entries (no bank conflicts); since (R_s - 1) NS_s = NS_{s+1} - NS_s the stages follow each other
// and the table has L - r_0 entries.
template <class PL, typename C>
__device__ __forceinline__ void stage_twiddles(C* tab, const C* __restrict__ tw, int tid, int nthr) {
  constexpr int L = PL::L, R0 = PL::r(0);
  for (int j = tid; j < L - R0; j += nthr) {
    int ns = R0, st = 1;
    while (st + 1 < PL::n && j >= ns * PL::r(st) - R0) {
      ns *= PL::r(st);
      ++st;
    }
    const int i = j - (ns - R0);
    const int m = i / ns + 1, kk = i - (m - 1) * ns;
    tab[j] = __ldg(tw + kk * m * (L / (ns * PL::r(st))));
  }
}
// twiddle m of butterfly kk in the stage with NS and step: from the per-stage table in shared
// memory (TWS), or from the plain table through the read-only path
template <bool TWS, class PL, int NS, typename C>
__device__ __forceinline__ C stage_tw(const C* __restrict__ tw, int m, int kk, int step) {
  if constexpr (TWS) return tw[(NS - PL::r(0)) + (m - 1) * NS + kk];
  else return __ldg(tw + kk * m * step);
}

// twiddle i of the table: from global memory through the read-only path, or (TWS) from a copy
// of the table in shared memory
template <bool TWS, typename C> __device__ __forceinline__ C tw_load(const C* __restrict__ tw, int i) {
  if constexpr (TWS) {
    return tw[i];
  } else {
    return __ldg(tw + i);
  }
}

// Twiddles and DFT of one butterfly; output m to put(m, value).
template <class PL, int R, int NS, bool INV, bool TWS, typename C, class Put>
__device__ __forceinline__ void butterfly(C (&v)[R], const C* __restrict__ tw, int kk, int step, const Put& put) {
  if constexpr (PL::two_float && INV && sizeof(C) == 8) {
    cdf d[R];
    d[0] = widen(v[0]);
#pragma unroll
    for (int m = 1; m < R; ++m) {
      d[m] = widen(v[m]);
      if (NS > 1) {
        C w = stage_tw<TWS, PL, NS>(tw, m, kk, step);
        w.y = -w.y;
        d[m] = cmul(d[m], widen(w));
      }
    }
    Dft<R, INV, cdf>::run(d);
#pragma unroll
    for (int m = 0; m < R; ++m) put(m, narrow(d[m]));
  } else {
    if (NS > 1) {
#pragma unroll
      for (int m = 1; m < R; ++m) {
        C w = stage_tw<TWS, PL, NS>(tw, m, kk, step);
        if (INV) w.y = -w.y;
        v[m] = cmul(v[m], w);
      }
    }
    Dft<R, INV, C>::run(v);
#pragma unroll
    for (int m = 0; m < R; ++m) put(m, v[m]);
  }
}

// one stage on rows; element e of sequence s at buf[s * pitch + at(e)]
template <class PL, int R, int NS, bool INV, bool TWS = false, typename C>
__device__ __forceinline__ void stage_fixed(C* buf, int s, int t, bool active, const C* __restrict__ tw, bool wsync) {
  constexpr int L = PL::L, T = PL::T;
  using P = RowPos<L>;
  constexpr int nb = L / R;
  constexpr int KB = (nb + T - 1) / T;
  constexpr bool EXACT = nb % T == 0;
  constexpr int step = L / (NS * R);
  // power-of-two lengths: the stores' pq NS R + kk + m NS splits into disjoint parts too
  const int tin = P::at(t);
  const int tout = P::pow2 ? P::at(stockham_out<NS, R>(t)) : 0;
  C v[KB][R];
  C* sb = buf + s * P::pitch;
  if (active) {
#pragma unroll
    for (int k = 0; k < KB; ++k)
      if (EXACT || t + k * T < nb) {
#pragma unroll
        for (int m = 0; m < R; ++m)
          v[k][m] = sb[EXACT ? row_join<L>(tin, P::at(k * T + m * nb)) : P::at(t + k * T + m * nb)];
      }
  }
  if (wsync) __syncwarp(); else __syncthreads();
  if (active) {
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int b = t + k * T;
      if (!EXACT && b >= nb) continue;
      const int base = stockham_out<NS, R>(b);
      butterfly<PL, R, NS, INV, TWS>(v[k], tw, b % NS, step, [&](int m, C x) {
        if constexpr (P::pow2) sb[tout ^ P::at((k * T / NS) * (NS * R) + (k * T) % NS + m * NS)] = x;
        else sb[P::at(base + m * NS)] = x;
      });
    }
  }
  if (wsync) __syncwarp(); else __syncthreads();
}

template <class PL, int ST, int NS, bool INV, bool TWS = false, typename C>
__device__ __forceinline__ void stages_fixed(C* buf, int s, int t, bool active, const C* __restrict__ tw,
                                             bool wsync) {
  if constexpr (ST < PL::n) {
    constexpr int R = PL::r(ST);
    stage_fixed<PL, R, NS, INV, TWS>(buf, s, t, active, tw, wsync);
    stages_fixed<PL, ST + 1, NS * R, INV, TWS>(buf, s, t, active, tw, wsync);
  }
}

// Row FFTs of a compile-time plan, sequence s by threads s T .. s T + T - 1 (RowPos layout).  TWS: tw
// points to the plan's per-stage twiddle table in shared memory (stage_twiddles).
template <class PL, bool INV, bool TWS = false, typename C>
__device__ __forceinline__ void fft_rows_fixed(C* buf, int nseq, const C* __restrict__ tw, int tid, int nthreads) {
  constexpr int T = PL::T;
  const int G = nthreads / T;
  const bool wsync = T <= 32 && (32 % T) == 0 && (nthreads % 32) == 0;
  for (int g0 = 0; g0 < nseq; g0 += G) {
    const int sl = tid / T, t = tid % T;
    const int s = g0 + sl;
    stages_fixed<PL, 0, 1, INV, TWS>(buf, s, t, sl < G && s < nseq, tw, wsync);
  }
}


// ---------------------------------------------------------------------------
// Column-tile FFTs with global-memory ends: sequence s = c * CT + col (c the
// field component, col the column in the tile) is column col of component c,
// element e of it lives at g[c * cstride + col + e * rstride] in global memory
// and at sm[e * W + s] in the shared tile.  IN_G: the first stage reads its
// butterfly inputs from global memory (columns >= ccols read as zero); OUT_G:
// the last stage writes its outputs to global memory (columns < ncol only).
// Every other stage goes through the shared tile.
// ---------------------------------------------------------------------------
template <typename C> struct ColIO {
  const C* gin;
  C* gout;
  size_t cstride, rstride;
  int ccols, ncol;
};

template <class PL, int R, int NS, int W, int CT, bool INV, bool FROM_G, bool TO_G, bool TWS = false, typename C>
__device__ __forceinline__ void stage_col(C* sm, const ColIO<C>& io, int s, int t, bool active,
                                          const C* __restrict__ tw) {
  constexpr int L = PL::L, T = PL::T;
  constexpr int nb = L / R;
  constexpr int KB = (nb + T - 1) / T;
  constexpr bool EXACT = nb % T == 0;
  constexpr int step = L / (NS * R);
  const int c = s / CT, col = s - c * CT;
  C v[KB][R];
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = t + k * T;
    if (active && (EXACT || b < nb)) {
      if (FROM_G) {
        const C* gp = io.gin + c * io.cstride + col;
        const bool ok = col < io.ccols;
#pragma unroll
        for (int m = 0; m < R; ++m) {
          const int e = b + m * nb;
          v[k][m] = ok ? gp[(size_t)e * io.rstride] : cmk<C>(0, 0);
        }
      } else {
#pragma unroll
        for (int m = 0; m < R; ++m) v[k][m] = sm[(b + m * nb) * W + s];
      }
    }
  }
  if (!FROM_G) __syncthreads();
  C* const gp = TO_G ? io.gout + c * io.cstride + col : nullptr;
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = t + k * T;
    if (active && (EXACT || b < nb) && (!TO_G || col < io.ncol)) {
      const int base = stockham_out<NS, R>(b);
      butterfly<PL, R, NS, INV, TWS>(v[k], tw, b % NS, step, [&](int m, C x) {
        if constexpr (TO_G) gp[(size_t)(base + m * NS) * io.rstride] = x;
        else sm[(base + m * NS) * W + s] = x;
      });
    }
  }
  if (!TO_G) __syncthreads();
}

template <class PL, int ST, int NS, int W, int CT, bool INV, bool IN_G, bool OUT_G, bool TWS = false, typename C>
__device__ __forceinline__ void stages_col(C* sm, const ColIO<C>& io, int s, int t, bool active,
                                           const C* __restrict__ tw) {
  if constexpr (ST < PL::n) {
    constexpr int R = PL::r(ST);
    constexpr bool FIRST = (ST == 0), LAST = (ST + 1 == PL::n);
    stage_col<PL, R, NS, W, CT, INV, IN_G && FIRST, OUT_G && LAST, TWS>(sm, io, s, t, active, tw);
    stages_col<PL, ST + 1, NS * R, W, CT, INV, IN_G, OUT_G, TWS>(sm, io, s, t, active, tw);
  }
}

// FFT of the W = 3 * CT columns of a tile; lanes walk across columns (COLMAP).
// TWS: tw points to the plan's per-stage twiddle table in shared memory (stage_twiddles).
template <class PL, int W, int CT, bool INV, bool IN_G, bool OUT_G, bool TWS = false, typename C>
__device__ __forceinline__ void fft_col_fixed(C* sm, const ColIO<C>& io, const C* __restrict__ tw, int tid,
                                              int nthreads) {
  constexpr int T = PL::T;
  const int G = nthreads / T;
  for (int g0 = 0; g0 < W; g0 += G) {
    const int sl = tid % G, t = tid / G;
    const int s = g0 + sl;
    const bool active = t < T && s < W;
    stages_col<PL, 0, 1, W, CT, INV, IN_G, OUT_G, TWS>(sm, io, s, t, active, tw);
  }
}

}  // namespace hs
