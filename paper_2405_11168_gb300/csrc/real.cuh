// Real-space pass of the basic scheme on a real displacement field: strain stencil, constitutive
// step and adjoint stencil, marching along z (FP32 iterations and FP64 sweeps; the contract is
// k_march's, see march.cuh for the plane and row conventions).
//
// Sum/difference form.  With s_x, s_y, s_z = +1 for the upper and -1 for the lower corner along an
// axis, T1 holds the corners with s_x s_y s_z = +1 and T2 the others (Eqs. DA1, DA2), so on T1
// s_x = s_y s_z and on T2 s_x = -s_y s_z.  The two gradients therefore are
//   4 D^T1_x u = W_x + H_x,   4 D^T2_x u = W_x - H_x   (y, z alike),
//   W_x = sum over 8 corners of s_x u,   H_x = sum over 8 corners of s_y s_z u,
// and the 6 sums of a component come from three stages of sums and differences (z, x, y), of which
// the first is shared by four voxels and the second by two: 12 additions per component and voxel
// where the two tetrahedra taken apart need 14.  Strain and stress are linear, so the law is
// applied to the pair (4E + W, H), and sigma^T1, sigma^T2 = (W +- H) / 4.  The mean stress and the
// fields need the W half alone.  The adjoint runs the stages backwards (y, z, x): a voxel row
// leaves 4 numbers per component, a corner row 2, of which one crosses to the column on the left
// (one shuffle per component and corner row; taken apart, two to four).  17 additions per
// component instead of 20.  Strains are formed as 4 times, forces would come out as 16 times their
// value; the phase tables hold the stiffness divided by 16 (kTabScale), exactly, so no factor is left.
//
// Pairs.  (W, H) of a strain or stress component travel as one two-lane value: f32x2 instructions
// in FP32, two scalars in FP64.  The stages keep DS = (difference along x, sum along z) with SD
// and SS with DD, which gives every y stage as one packed operation; the z derivatives come out
// with the lanes exchanged, (H, W), which is the order in which the adjoint wants them.
//
// Bounds: FP32 by instruction issue, FP64 by the FP64 pipe (2 lanes per SM and clock).
#pragma once
#include "march.cuh"

namespace hs {

enum { REAL_BULK = 1, REAL_SRC = 2, REAL_EIGEN = 4, REAL_SPLIT = 8 };

template <typename T> struct Pair;  // two-lane arithmetic, every operation rounded lane by lane
template <> struct Pair<float> {
  using V = float2;
  static __device__ __forceinline__ V mk(float x, float y) { return make_float2(x, y); }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
  // b * +-1 is exact, so these are rounded sums and differences
  static __device__ __forceinline__ V addsub(V a, V b) { return __ffma2_rn(b, make_float2(1.f, -1.f), a); }
  static __device__ __forceinline__ V subadd(V a, V b) { return __ffma2_rn(b, make_float2(-1.f, 1.f), a); }
};
template <> struct Pair<double> {
  using V = double2;
  static __device__ __forceinline__ V mk(double x, double y) { return make_double2(x, y); }
  static __device__ __forceinline__ V add(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ V mul(V a, V b) { return make_double2(a.x * b.x, a.y * b.y); }
  static __device__ __forceinline__ V fma(V a, V b, V c) {
    return make_double2(::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y));
  }
  static __device__ __forceinline__ V addsub(V a, V b) { return make_double2(a.x + b.x, a.y - b.y); }
  static __device__ __forceinline__ V subadd(V a, V b) { return make_double2(a.x - b.x, a.y + b.y); }
};

// Constitutive laws on (W, H) pairs of the engineering strain; index 2 (the zz component) has its
// lanes exchanged on both sides.
template <typename T> struct RealIso {
  using V = typename Pair<T>::V;
  const T* tab;
  __device__ __forceinline__ void stress(int ph, const V (&e)[6], V (&s)[6]) const {
    using P = Pair<T>;
    V lam, mu;
    iso_pairs(tab, ph, lam, mu);
    const V m2 = P::add(mu, mu);
    V tr = P::add(e[0], e[1]);
    tr = P::mk(tr.x + e[2].y, tr.y + e[2].x);
    const V lt = P::mul(lam, tr);
    s[0] = P::fma(m2, e[0], lt);
    s[1] = P::fma(m2, e[1], lt);
    s[2] = P::fma(m2, e[2], P::mk(lt.y, lt.x));
    s[3] = P::mul(mu, e[3]);
    s[4] = P::mul(mu, e[4]);
    s[5] = P::mul(mu, e[5]);
  }
};
template <typename T> struct RealAniso {
  using V = typename Pair<T>::V;
  const T* tab;
  __device__ __forceinline__ void stress(int ph, const V (&e)[6], V (&s)[6]) const {
    constexpr int ST = kAnisoStride<T>;
    using L = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int NL = 16 / (int)sizeof(T);
    const L* c = reinterpret_cast<const L*>(tab + (size_t)ST * ph);
    T C[ST];
#pragma unroll
    for (int i = 0; i < ST / NL; ++i) {
      const L v = __ldg(c + i);
      const T* w = reinterpret_cast<const T*>(&v);
#pragma unroll
      for (int j = 0; j < NL; ++j) C[i * NL + j] = w[j];
    }
    const T w[6] = {e[0].x, e[1].x, e[2].y, e[3].x, e[4].x, e[5].x};
    const T h[6] = {e[0].y, e[1].y, e[2].x, e[3].y, e[4].y, e[5].y};
    T sw[6], sh[6];
    int k = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i; j < 6; ++j, ++k) {
        // row i = 0 initialises every entry
        if (i == 0) {
          if (j == 0) {
            sw[0] = C[0] * w[0];
            sh[0] = C[0] * h[0];
          } else {
            sw[0] = ::fma(C[j], w[j], sw[0]);
            sh[0] = ::fma(C[j], h[j], sh[0]);
            sw[j] = C[j] * w[0];
            sh[j] = C[j] * h[0];
          }
        } else {
          sw[i] = ::fma(C[k], w[j], sw[i]);
          sh[i] = ::fma(C[k], h[j], sh[i]);
          if (j != i) {
            sw[j] = ::fma(C[k], w[i], sw[j]);
            sh[j] = ::fma(C[k], h[i], sh[j]);
          }
        }
      }
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] = i == 2 ? Pair<T>::mk(sh[i], sw[i]) : Pair<T>::mk(sw[i], sh[i]);
  }
};

constexpr int kSumBytes = 56;  // RealSums, per thread: three float4 (two high parts, two low parts), one float2

// Shared memory of k_real.  xp: row pitch (elements); host and device use the same function.
struct RealLayout {
  size_t ring, ids, src, edge, red, bar, total;
};
__host__ __device__ inline RealLayout real_layout(int xp, int nthr, int ty, bool has_src, int tsize) {
  RealLayout L;
  const int NR = ty + 2;
  size_t off = 0;
  L.ring = off;  // [3 planes][3 components][NR][xp]
  off += hs_align16((size_t)tsize * 3 * 3 * NR * xp);
  L.ids = off;   // [2][ty + 1][xp]
  off += hs_align16((size_t)2 * 2 * (ty + 1) * xp);
  L.src = off;   // [3][3 components][ty][xp]
  off += hs_align16(has_src ? (size_t)4 * 3 * 3 * ty * xp : 0);
  L.edge = off;  // [2][nwarps][ty][3] x (own, left)
  off += hs_align16((size_t)2 * 2 * tsize * (nthr / 32) * ty * 3);
  L.red = off;   // block sums; FP32: before them the threads' running sums (RealSums)
  off += tsize == 4 && (size_t)kSumBytes * nthr > kReduceScratch ? (size_t)kSumBytes * nthr : kReduceScratch;
  L.bar = off;
  off += 32;
  L.total = off;
  return L;
}

// A thread's running sums of the FP32 pass, 6 stress components and |F|^2, in shared memory as unevaluated
// pairs (high, low) of floats.  FP32 registers hold the terms of a few planes only (MarchArgs::sum_planes)
// and are then added here, the rounding error of each addition kept in the low part (Knuth's two-sum), so a
// sum's accuracy does not depend on the chunk.  One FP32 chain over a whole chunk (32 planes of 4 rows at 192^3)
// left up to 1.7e-6 in the mean stress of a uniform field.
struct RealSums {
  using P = Pair<float>;
  float4* s;  // [3][nthr]
  float2* f;  // [nthr]
  __device__ __forceinline__ RealSums(unsigned char* base, int tid, int nthr)
      : s(reinterpret_cast<float4*>(base) + tid), f(reinterpret_cast<float2*>(base + (size_t)48 * nthr) + tid) {}
  __device__ __forceinline__ void clear(int nthr) const {
#pragma unroll
    for (int i = 0; i < 3; ++i) s[i * nthr] = make_float4(0.f, 0.f, 0.f, 0.f);
    *f = make_float2(0.f, 0.f);
  }
  // the registers' sums go in and start again from 0
  __device__ __forceinline__ void take(float (&sacc)[6], float& facc, int nthr) const {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float4 v = s[i * nthr];
      two_sum(v, make_float2(sacc[2 * i], sacc[2 * i + 1]));
      s[i * nthr] = v;
      sacc[2 * i] = sacc[2 * i + 1] = 0.f;
    }
    float4 v = make_float4(f->x, 0.f, f->y, 0.f);
    two_sum(v, make_float2(facc, 0.f));
    *f = make_float2(v.x, v.z);
    facc = 0.f;
  }
  // (v.x, v.y) + b with the rounding errors added to (v.z, v.w)
  static __device__ __forceinline__ void two_sum(float4& v, float2 b) {
    auto sub = [](float2 a, float2 c) { return __ffma2_rn(c, make_float2(-1.f, -1.f), a); };
    const float2 hi = make_float2(v.x, v.y), t = P::add(hi, b), z = sub(t, hi);
    const float2 lo = P::add(P::add(sub(hi, sub(t, z)), sub(b, z)), make_float2(v.z, v.w));
    v = make_float4(t.x, t.y, lo.x, lo.y);
  }
  // a warp's sums (lane l: value l / 4): the high parts in FP64, the low parts, which are 2^-24 of them, in FP32
  // (an FP64 conversion costs a warp 64 cycles).  An infinite high part has no low part.
  __device__ __forceinline__ double warp_total(bool xact, int nthr) const {
    double h[8];
    float l[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = i < 3 ? s[i * nthr] : make_float4(f->x, 0.f, f->y, 0.f);
      const bool in = xact || i == 3;
      h[2 * i] = in ? (double)v.x : 0.0;
      h[2 * i + 1] = in && i < 3 ? (double)v.y : 0.0;
      l[2 * i] = in && v.z == v.z ? v.z : 0.f;
      l[2 * i + 1] = in && i < 3 && v.w == v.w ? v.w : 0.f;
    }
    const double scale = (threadIdx.x & 31) < 24 ? 0.5 / (double)kTabScale<float> : 1.0;
    return scale * (warp_sum8(h) + (double)warp_sum8(l));
  }
};

// Copy of one plane by warp 0: u rows y0 - 1 .. y0 + TY of corner plane pu into ring slot `slot`, the id
// rows y0 .. y0 + TY of voxel plane pu into ids buffer ib (ib < 0: none), the source rows of output
// plane ps into source buffer sb (sb < 0: none), as bulk copies that complete on bar.  Rows of a
// component that follow each other both in global memory and in the ring go in one copy (at most
// three where y wraps), issued by one lane per component; otherwise every lane copies single rows.
template <typename T, int TY>
__device__ __forceinline__ void real_prefetch_bulk(const MarchArgs<T>& a, const RealLayout& lay, unsigned char* sm,
                                                   int xp, int y0, int pu, int slot, int ib, int ps, int sb,
                                                   uint64_t* bar) {
  constexpr int NR = TY + 2;
  const int n1 = a.n1, n2 = a.n2, n3 = a.n3, lane = threadIdx.x & 31;
  const size_t rplane = (size_t)n2 * n1, rcomp = (size_t)n3 * rplane;
  const int gz = pu < 0 ? pu + n3 : (pu >= n3 ? pu - n3 : pu);
  const int zs = ps >= n3 ? ps - n3 : ps;
  const int nu = 3 * NR, ni = ib >= 0 ? TY + 1 : 0, ns = sb >= 0 ? 3 * TY : 0;
  if (lane == 0)
    mbar_arrive_expect_tx(bar, (unsigned)(((size_t)nu * sizeof(T) + (size_t)ni * 2 + (size_t)ns * 4) * n1));
  __syncwarp();
  auto copy = [&](void* dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
  };
  T* const ru = reinterpret_cast<T*>(sm + lay.ring) + (size_t)slot * nu * xp;
  uint16_t* const ri = reinterpret_cast<uint16_t*>(sm + lay.ids) + (size_t)ib * (TY + 1) * xp;
  float* const rs = reinterpret_cast<float*>(sm + lay.src) + (size_t)sb * ns * xp;
  if (xp == n1) {
    // lanes 0-2: u components; 3: ids; 4-6: source components
    const int c = lane < 3 ? lane : lane - 4;
    int y, rows, esz;
    unsigned char* dst;
    const unsigned char* plane;
    if (lane < 3) {
      y = y0 - 1; rows = NR; esz = (int)sizeof(T);
      dst = reinterpret_cast<unsigned char*>(ru + (size_t)c * NR * xp);
      plane = reinterpret_cast<const unsigned char*>(a.ureal + c * rcomp + (size_t)gz * rplane);
    } else if (lane == 3) {
      y = y0; rows = ni; esz = 2;
      dst = reinterpret_cast<unsigned char*>(ri);
      plane = reinterpret_cast<const unsigned char*>(a.ids + (size_t)gz * rplane);
    } else {
      y = y0; rows = (lane < 7 && ns > 0) ? TY : 0; esz = 4;
      dst = reinterpret_cast<unsigned char*>(rs + (size_t)c * TY * xp);
      plane = reinterpret_cast<const unsigned char*>(a.src + c * rcomp + (size_t)zs * rplane);
    }
    if (y < 0) y += n2;
    const unsigned rowbytes = (unsigned)(n1 * esz);
    for (int r = 0; r < rows;) {
      const int run = min(rows - r, n2 - y);
      copy(dst + (size_t)r * rowbytes, plane + (size_t)y * rowbytes, (unsigned)run * rowbytes);
      r += run;
      y = 0;
    }
  } else {
    for (int i = lane; i < nu + ni + ns; i += 32) {
      if (i < nu) {
        const int c = i / NR, gy = (y0 - 1 + (i - c * NR) + n2) % n2;
        copy(ru + (size_t)i * xp, a.ureal + c * rcomp + (size_t)gz * rplane + (size_t)gy * n1, (unsigned)(n1 * sizeof(T)));
      } else if (i < nu + ni) {
        const int r = i - nu, gy = (y0 + r) % n2;
        copy(ri + (size_t)r * xp, a.ids + (size_t)gz * rplane + (size_t)gy * n1, (unsigned)(n1 * 2));
      } else {
        const int r = i - nu - ni, c = r / TY, gy = (y0 + (r - c * TY)) % n2;
        copy(rs + (size_t)r * xp, a.src + c * rcomp + (size_t)zs * rplane + (size_t)gy * n1, (unsigned)(n1 * 4));
      }
    }
  }
}

// The same for half a row (REAL_SPLIT): columns x0 .. x0 + nx - 1 from position 2 of a ring row on, the two columns
// on their left before them (periodic), ids of the block's columns.  x0 is 0 or a multiple of 8.
template <typename T, int TY>
__device__ __forceinline__ void real_prefetch_half(const MarchArgs<T>& a, const RealLayout& lay, unsigned char* sm,
                                                   int xp, int x0, int nx, int y0, int pu, int slot, int ib, uint64_t* bar) {
  constexpr int NR = TY + 2;
  const int n1 = a.n1, n2 = a.n2, n3 = a.n3, lane = threadIdx.x & 31;
  const size_t rplane = (size_t)n2 * n1, rcomp = (size_t)n3 * rplane;
  const int gz = pu < 0 ? pu + n3 : (pu >= n3 ? pu - n3 : pu);
  const int nu = 3 * NR, ni = ib >= 0 ? TY + 1 : 0;
  if (lane == 0) mbar_arrive_expect_tx(bar, (unsigned)(nu * (nx + 2) * sizeof(T) + ni * nx * 2));
  __syncwarp();
  auto copy = [&](void* dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
  };
  T* const ru = reinterpret_cast<T*>(sm + lay.ring) + (size_t)slot * nu * xp;
  uint16_t* const ri = reinterpret_cast<uint16_t*>(sm + lay.ids) + (size_t)ib * (TY + 1) * xp;
  for (int i = lane; i < nu + ni; i += 32) {
    if (i < nu) {
      const int c = i / NR, gy = (y0 - 1 + (i - c * NR) + n2) % n2;
      const T* const row = a.ureal + c * rcomp + (size_t)gz * rplane + (size_t)gy * n1;
      T* const d = ru + (size_t)i * xp;
      if (x0 > 0) {
        copy(d, row + x0 - 2, (unsigned)((nx + 2) * sizeof(T)));
      } else {
        copy(d, row + n1 - 2, (unsigned)(2 * sizeof(T)));
        copy(d + 2, row, (unsigned)(nx * sizeof(T)));
      }
    } else {
      const int r = i - nu, gy = (y0 + r) % n2;
      copy(ri + (size_t)r * xp, a.ids + (size_t)gz * rplane + (size_t)gy * n1 + x0, (unsigned)(nx * 2));
    }
  }
}

// Barrier of the two blocks of a cluster, with the shared-memory writes before it visible to both after it; a
// word of the other block's shared memory.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned peer_addr(const void* p, int peer) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(p)), "r"(peer));
  return a;
}
__device__ __forceinline__ double peer_load(const double* p, int peer) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(v) : "r"(peer_addr(p, peer)) : "memory");
  return v;
}
__device__ __forceinline__ int peer_load(const int* p, int peer) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];\n" : "=r"(v) : "r"(peer_addr(p, peer)) : "memory");
  return v;
}

// Rows of n elements of E bytes by the block's warps, one row per warp and turn: cp.async in the widest chunks
// (16, 8 or 4 bytes) that start and end every row; 2-byte rows that do not start on 4 bytes element by element.
// Every thread over every row in turn, 8 bytes at a time, left most of a block without a copy; rows per warp and the
// compile-time pitch: FP32 force pass 60.8 -> 33.7 us at 100^3, 102 -> 65.7 at 126 x 90 x 210, 254 -> 189
// at 220 x 200 x 180.
template <typename E, class Src, class Dst>
__device__ __forceinline__ void rows_async(int nrows, int n, const Src& src, const Dst& dst) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned bytes = (unsigned)(n * sizeof(E));
  for (int r = warp; r < nrows; r += nw) {
    const unsigned char* const s = reinterpret_cast<const unsigned char*>(src(r));
    unsigned char* const d = reinterpret_cast<unsigned char*>(dst(r));
    const unsigned d0 = smem_u32(d), a = bytes | (unsigned)reinterpret_cast<uintptr_t>(s);
    if ((a & 15) == 0) {
      for (unsigned q = 16 * lane; q < bytes; q += 512) cp_async16(d + q, s + q);
    } else if ((a & 7) == 0) {
      for (unsigned q = 8 * lane; q < bytes; q += 256)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d0 + q), "l"(s + q) : "memory");
    } else if ((a & 3) == 0) {
      for (unsigned q = 4 * lane; q < bytes; q += 128)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d0 + q), "l"(s + q) : "memory");
    } else {
      for (int q = lane; q < n; q += 32) reinterpret_cast<E*>(d)[q] = reinterpret_cast<const E*>(s)[q];
    }
  }
}

// The same plane by every warp, for rows that bulk copies cannot take (a.bulk = 0).  Ends with a commit.
template <typename T, int TY>
__device__ __forceinline__ void real_prefetch_async(const MarchArgs<T>& a, const RealLayout& lay, unsigned char* sm,
                                                    int xp, int y0, int pu, int slot, int ib, int ps, int sb) {
  constexpr int NR = TY + 2;
  const int n1 = a.n1, n2 = a.n2, n3 = a.n3;
  const size_t rplane = (size_t)n2 * n1, rcomp = (size_t)n3 * rplane;
  const int gz = pu < 0 ? pu + n3 : (pu >= n3 ? pu - n3 : pu);
  T* const ru = reinterpret_cast<T*>(sm + lay.ring) + (size_t)slot * 3 * NR * xp;
  const T* const u = a.ureal + (size_t)gz * rplane;
  rows_async<T>(3 * NR, n1,
                [&](int r) {
                  const int c = r / NR, gy = (y0 - 1 + (r - c * NR) + n2) % n2;
                  return u + c * rcomp + (size_t)gy * n1;
                },
                [&](int r) { return ru + r * xp; });
  if (ib >= 0) {
    uint16_t* const ri = reinterpret_cast<uint16_t*>(sm + lay.ids) + (size_t)ib * (TY + 1) * xp;
    const uint16_t* const ids = a.ids + (size_t)gz * rplane;
    rows_async<uint16_t>(TY + 1, n1, [&](int r) { return ids + (size_t)((y0 + r) % n2) * n1; },
                         [&](int r) { return ri + r * xp; });
  }
  if (sb >= 0) {
    const int zs = ps >= n3 ? ps - n3 : ps;
    float* const rs = reinterpret_cast<float*>(sm + lay.src) + (size_t)sb * 3 * TY * xp;
    const float* const src = a.src + (size_t)zs * rplane;
    rows_async<float>(3 * TY, n1,
                      [&](int r) {
                        const int c = r / TY;
                        return src + c * rcomp + (size_t)((y0 + (r - c * TY)) % n2) * n1;
                      },
                      [&](int r) { return rs + r * xp; });
  }
  cp_async_commit();
}

// Resident blocks per SM that the registers of an FP32 pass with bulk copies must allow: 16 warps, 12 for blocks of up
// to 128 threads, whose values then all stay in (up to 168) registers.  16 for those too: 128^3 34.6 -> 30.9 us, but
// 64^3 14.4 -> 15.0, 96 x 192 x 384 95.5 -> 98.5, 64 x 256 x 256 48.1 -> 51.6.  0: left to the compiler.
__host__ __device__ constexpr int real_min_blocks(int nt, bool bulk) { return !bulk ? 0 : nt >= 256 ? 512 / nt : 384 / nt; }

// One block: corner rows y0 .. y0 + TY - 1 (TY divides N2) of one z chunk, thread x <-> column x.
// XP > 0: compile-time row pitch in shared memory (N1 <= XP), so that row offsets are immediates;
// XP = 0: a.xp.  NT: the largest block (its registers).  OPT: what the launch has, as compile-time
// facts (tested at run time they cost a fifth of the instructions: 157.9 against 125.6 M per launch at
// 256^3, 0.232 against 0.187 ms): REAL_BULK planes by bulk copies (XP = 0: a.bulk decides), REAL_SRC a
// correction source (else none), REAL_EIGEN an eigenstress (else none).  BATCH: grid.z items, every workspace pointer
// moved per item; a single solve's launch uses the arguments as they come.
//
// A step handles voxel plane p between corner planes p - 1 and p (ring slots filled two steps ahead)
// and completes corner plane p - 1.  One block barrier per step: it publishes the left-going sums of
// each warp's first column, which the previous warp's last column needs, and frees ring slot p - 2.
//
// FP32 sums: sacc and facc hold the terms of sum_planes planes, then RealSums takes them.  The groups are a loop
// around the steps; the same addition behind a test in each step cost the whole pass 11% (256^3: 174 -> 194 us, nested 175),
// because the compiler then kept the sums and the test live through the step.
//
// REAL_SPLIT (FP64, more than 256 columns): the two blocks of a cluster take half the columns each, the barrier
// of a step is the cluster's, and a half's last column reads the sums of the other half's first one from
// that block's shared memory.  One block of 512 threads has 128 registers and shared memory for tiles of 2
// rows, which compute 3 voxel rows for 2; halves of 256 run 8 rows with 255 registers: FP64 sweep of 512^3, 21-constant
// law, 64.1 -> 51.6 ms.
template <typename T, int TY, class MAT, int MODE, int XP, int NT, int OPT, bool BATCH>
__global__ void __launch_bounds__(NT, real_min_blocks(NT, (OPT & REAL_BULK) != 0)) k_real(const MarchArgs<T> a_, const MAT mat_) {
  using P = Pair<T>;
  using V = typename P::V;
  constexpr int NR = TY + 2;
  constexpr bool F64 = sizeof(T) == 8;
  constexpr bool SPLIT = (OPT & REAL_SPLIT) != 0;
  constexpr bool FORCE = MODE == MODE_FORCE || MODE == MODE_FORCE_FIELDS;
  constexpr bool FIELDS = MODE == MODE_FIELDS || MODE == MODE_FORCE_FIELDS;
  const MarchArgs<T> a = BATCH ? march_item_args(a_) : a_;
  MAT mat = mat_;
  if (BATCH) mat.tab = a.mat;
  bool skip = false;
  if constexpr (SPLIT) skip = a.st->retired || (a.skip_if_done && a.st->done);
  else if (a.st->retired || (a.skip_if_done && a.st->done)) return;
  extern __shared__ __align__(128) unsigned char smraw[];
  const int n1 = a.n1, n2 = a.n2, n3 = a.n3;
  const int xp = XP > 0 ? XP : a.xp;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nthr >> 5;
  constexpr int XO = SPLIT ? 2 : 0;  // position of the block's first column in a ring row
  const int half = SPLIT ? (int)(blockIdx.x & 1) : 0;  // also the rank in the cluster
  const int nx = SPLIT ? n1 >> 1 : n1, x0 = SPLIT ? half * nx : 0;  // columns of the block
  const int y0 = (SPLIT ? blockIdx.x >> 1 : blockIdx.x) * TY;
  const int z0 = blockIdx.y * a.zc;
  const int zc = min(a.zc, n3 - z0);
  const size_t rplane = (size_t)n2 * n1, rcomp = (size_t)n3 * rplane;
  constexpr bool has_src = FORCE && (OPT & REAL_SRC) != 0;
  const bool bulk = SPLIT || (OPT & REAL_BULK) != 0 || (XP == 0 && a.bulk != 0);

  const RealLayout lay = real_layout(xp, nthr, TY, has_src, (int)sizeof(T));
  const T* const ring = reinterpret_cast<const T*>(smraw + lay.ring);
  const uint16_t* const sids = reinterpret_cast<const uint16_t*>(smraw + lay.ids);
  const float* const ssrc = reinterpret_cast<const float*>(smraw + lay.src);
  V* const edge = reinterpret_cast<V*>(smraw + lay.edge);  // [2][nw][TY][3]: (own part of the receiver, left of the sender)
  uint64_t* const bar = reinterpret_cast<uint64_t*>(smraw + lay.bar);

  if constexpr (SPLIT) {
    // both blocks run or neither does: a block does not read the memory of one that has left
    int* const flag = reinterpret_cast<int*>(smraw + lay.red);
    if (tid == 0) *flag = skip ? 1 : 0;
    cluster_sync();
    const int leave = *flag | peer_load(flag, half ^ 1);
    cluster_sync();
    if (leave) return;
  }
  const int x = x0 + tid;
  const bool xact = tid < nx;
  const int xr = xact ? tid : 0;
  const int xmr = SPLIT ? xr + XO - 1 : xr == 0 ? n1 - 1 : xr - 1;
  const bool recv_shfl = lane < 31 && tid + 1 < nx;  // the column on the right sits in this warp
  // a warp's first column publishes its left-going sums, its last one its own sums (N1 is even, so
  // no lane is both)
  const bool at_edge = lane == 0 || (xact && !recv_shfl);
  const int edge_half = lane == 0 ? 1 : 0;

  V carry[TY][3];  // corner plane p: (own, left-going) sums of F from voxel plane p
#pragma unroll
  for (int r = 0; r < TY; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) carry[r][k] = P::mk(0, 0);
  T sacc[6];  // sum of 4 kTabScale sigma over the W half: 2 kTabScale (sigma^T1 + sigma^T2)
#pragma unroll
  for (int i = 0; i < 6; ++i) sacc[i] = 0;
  T facc = 0;
  constexpr bool SUMS = !F64 && FORCE;  // FP32: the sums of several planes are kept in RealSums
  const RealSums sums(smraw + lay.red, tid, nthr);
  if constexpr (SUMS) sums.clear(nthr);
  T E4[6];  // 4 x engineering macro strain
#pragma unroll
  for (int i = 0; i < 6; ++i) E4[i] = (i < 3 ? T(4) : T(8)) * macro_E(a, i);

  // output force: element size, bytes per component and row, byte offset of this column in corner plane p - 1
  const int fsz = (F64 && !a.fout_f32) ? 8 : 4;
  const int64_t fcomp = (int64_t)rcomp * fsz;
  const int frstep = n1 * fsz;
  int64_t fplane = ((int64_t)(z0 - 1) * (int64_t)rplane + (int64_t)y0 * n1 + x) * fsz;
  bool timed_out = false;
  auto prefetch = [&](int pu, bool want_ids) {
    const int q = pu - z0 + 1;  // plane pu sits in slot q % 3; step pu completes output plane pu - 1
    const int ib = want_ids ? (q & 1) : -1;
    const int sb = (has_src && pu > z0) ? q % 3 : -1;
    if (bulk) {
      if constexpr (SPLIT) {
        if (warp == 0) real_prefetch_half<T, TY>(a, lay, smraw, xp, x0, nx, y0, pu, q % 3, ib, bar + q % 3);
      } else if (warp == 0) real_prefetch_bulk<T, TY>(a, lay, smraw, xp, y0, pu, q % 3, ib, pu - 1, sb, bar + q % 3);
    } else {
      real_prefetch_async<T, TY>(a, lay, smraw, xp, y0, pu, q % 3, ib, pu - 1, sb);
    }
  };
  if (bulk) {
    if (tid == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) mbar_init(bar + q, 1);
      mbar_init_fence();
    }
    __syncthreads();  // the barriers are initialised before anyone waits on them
  }
  const int pend = FORCE ? z0 + zc : z0 + zc - 1;
  prefetch(z0 - 1, false);
  prefetch(z0, true);
  if (bulk) timed_out |= !mbar_wait(bar, 0);

  // steps in groups of sum_planes (FP32), after which the registers' sums move on
  const int group = SUMS ? a.sum_planes : pend - z0 + 1;
  auto group_end = [&]() {
    if constexpr (SUMS) sums.take(sacc, facc, nthr);
  };
  for (int p = z0; p <= pend; group_end())
  for (const int pe = min(p + group - 1, pend); p <= pe; ++p) {
    const int q = p - z0 + 1;
    const int sc = q % 3, sp = (q + 2) % 3;
    if (p < pend) {
      if (!bulk) {
        // the copies of plane p must be complete before the ring moves on
        cp_async_wait_all();
        __syncthreads();
      }
      prefetch(p + 1, true);
    }
    if (bulk) {
      timed_out |= !mbar_wait(bar + sc, (unsigned)((q / 3) & 1));
    } else if (p == pend) {
      cp_async_wait_all();
      __syncthreads();
    }
    const bool own_plane = p < z0 + zc;
    const bool out_plane = FORCE && p > z0;  // corner plane p - 1 belongs to this chunk
    const T* const rc = ring + sc * 3 * NR * xp;
    const T* const rp = ring + sp * 3 * NR * xp;
    const T* const rcx = rc + xr + XO;
    const T* const rpx = rp + xr + XO;
    const T* const rcl = rc + xmr;
    const T* const rpl = rp + xmr;
    const uint16_t* const idrow = sids + (q & 1) * (TY + 1) * xp + xr;
    const float* const srow = ssrc + sc * 3 * TY * xp + xr;
    V* const ed = edge + (q & 1) * nw * TY * 3;
    T* const my_edge = reinterpret_cast<T*>(ed + warp * TY * 3) + edge_half;
    // row 0 of corner plane p - 1, this column, component 0; moves on row by row
    unsigned char* frow = reinterpret_cast<unsigned char*>(a.fout) + fplane;
    fplane += (int64_t)rplane * fsz;
    const bool take = recv_shfl && out_plane, store = take && a.fout != nullptr;
    // FP64: lane l < 32 holds the z sums and differences of ring row l / 3, component l % 3 of the
    // column left of this warp's first (two additions per warp and plane instead of two per lane, row
    // and component); the other lanes' left columns come by shuffle
    T eS[2], eD[2];
    if constexpr (F64) {
      const int xl = SPLIT ? (warp << 5) + XO - 1 : ((warp << 5) + n1 - 1) % n1;
#pragma unroll
      for (int h = 0; h < (3 * NR + 31) / 32; ++h) {
        const int i = min(lane + 32 * h, 3 * NR - 1), o = ((i % 3) * NR + i / 3) * xp + xl;
        const T up = rc[o], um = rp[o];
        eS[h] = up + um;
        eD[h] = up - um;
      }
    }
    // (DS, SD) and (SS, DD) of ring row j
    auto stage_zx = [&](int j, V (&Pn)[3], V (&Qn)[3]) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int o = (c * NR + j) * xp;
        const T up = rcx[o], um = rpx[o];
        const V own = P::mk(up + um, up - um);
        V left;
        if constexpr (F64) {
          const int i = 3 * j + c;
          const T ls = __shfl_up_sync(0xffffffffu, own.x, 1), ld = __shfl_up_sync(0xffffffffu, own.y, 1);
          const T es = __shfl_sync(0xffffffffu, eS[i >> 5], i & 31), el = __shfl_sync(0xffffffffu, eD[i >> 5], i & 31);
          left = P::mk(lane == 0 ? es : ls, lane == 0 ? el : ld);
        } else {
          const T lu = rcl[o], lm = rpl[o];
          left = P::mk(lu + lm, lu - lm);
        }
        Pn[c] = P::subadd(own, left);
        Qn[c] = P::addsub(own, left);
      }
    };
    V Pn[3], Qn[3];
    stage_zx(0, Pn, Qn);
    V AP[3], AQ[3];  // (DS, SD) and (SS, DD) sums of the corner row being completed
#pragma unroll
    for (int jj = 1; jj <= TY + 1; ++jj) {
      if (!FORCE && jj == TY + 1) break;
      V Po[3], Qo[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) { Po[c] = Pn[c]; Qo[c] = Qn[c]; }
      stage_zx(jj, Pn, Qn);
      const int ph = idrow[(jj - 1) * xp];
      V e[6], s[6];
      {
        V gx[3], gy[3], gz[3];  // (W, H) of d/dx, d/dy; (H, W) of d/dz
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          gx[c] = P::addsub(Pn[c], Po[c]);
          gy[c] = P::subadd(Qn[c], Qo[c]);
          gz[c] = P::subadd(Pn[c], Po[c]);
        }
        e[0] = P::mk(gx[0].x + E4[0], gx[0].y);
        e[1] = P::mk(gy[1].x + E4[1], gy[1].y);
        e[2] = P::mk(gz[2].x, gz[2].y + E4[2]);
        e[3] = P::mk((gy[2].x + gz[1].y) + E4[3], gy[2].y + gz[1].x);
        e[4] = P::mk((gx[2].x + gz[0].y) + E4[4], gx[2].y + gz[0].x);
        e[5] = P::add(gx[1], gy[0]);
        e[5].x += E4[5];
      }
      mat.stress(ph, e, s);
      if (OPT & REAL_EIGEN) {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const T s0 = T(4) * kTabScale<T> * a.sig0[6 * ph + i];
          if (i == 2) s[i].y -= s0;
          else s[i].x -= s0;
        }
      }
      if (FIELDS) {
        if (jj <= TY && xact && own_plane) {  // the halo row belongs to the next tile
          const int pz = p >= n3 ? p - n3 : p;
          const size_t o = (size_t)pz * rplane + (size_t)(y0 + jj - 1) * n1 + x;
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            const T ev = (i == 2 ? e[i].y : e[i].x) * (i < 3 ? T(0.25) : T(0.125));
            const T sv = (i == 2 ? s[i].y : s[i].x) * (T(0.25) / kTabScale<T>);
            if (a.out_f32) {
              reinterpret_cast<float*>(a.eps_out)[i * rcomp + o] = (float)ev;
              reinterpret_cast<float*>(a.sig_out)[i * rcomp + o] = (float)sv;
            } else {
              reinterpret_cast<double*>(a.eps_out)[i * rcomp + o] = (double)ev;
              reinterpret_cast<double*>(a.sig_out)[i * rcomp + o] = (double)sv;
            }
          }
        }
      }
      if (!FORCE) continue;
      if (jj <= TY && own_plane) {
#pragma unroll
        for (int i = 0; i < 6; ++i) sacc[i] += (i == 2 ? s[i].y : s[i].x);
      }
      // adjoint: voxel row jj adds to corner rows jj - 1 (lower, completed here) and jj (upper)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const V sx = s[k == 0 ? 0 : (k == 1 ? 5 : 4)];
        const V sy = s[k == 0 ? 5 : (k == 1 ? 1 : 3)];
        const V szn = s[k == 0 ? 4 : (k == 1 ? 3 : 2)];
        const V sz = k == 2 ? szn : P::mk(szn.y, szn.x);  // (H, W)
        if (jj >= 2) {
          const int r = jj - 2;
          const V p1 = P::subadd(P::addsub(AP[k], sx), sz);
          const V q1 = P::subadd(AQ[k], sy);
          const V X = P::mk(q1.x + p1.x, q1.x - p1.x), Y = P::mk(q1.y + p1.y, q1.y - p1.y);
          const V f = P::subadd(P::add(carry[r][k], X), Y);  // corner plane p - 1: (own, left-going)
          carry[r][k] = P::addsub(X, Y);
          if (out_plane) {
            const T F0 = f.x + __shfl_down_sync(0xffffffffu, f.y, 1);
            if (at_edge) my_edge[(r * 3 + k) * 2] = edge_half ? f.y : f.x;
            const T F = has_src ? F0 + (T)srow[(k * TY + r) * xp] : F0;
            if (take) facc = ::fma(F, F, facc);
            if (store) {
              unsigned char* const fo = frow + k * fcomp;
              if (F64 && !a.fout_f32) *reinterpret_cast<double*>(fo) = (double)F;
              else *reinterpret_cast<float*>(fo) = (float)F;
            }
          }
        }
        AP[k] = P::add(sx, sz);
        AQ[k] = sy;
      }
      if (jj >= 2) frow += frstep;
    }
    if (SPLIT) cluster_sync(); else __syncthreads();
    if (out_plane) {
      // the last column of every warp: its own part and the left-going part of the column to its right
      for (int i = tid; i < nw * TY * 3; i += nthr) {
        const int k = i % 3, wr = i / 3, w = wr / TY, r = wr - w * TY;
        const int xe = min((w << 5) + 31, nx - 1);
        const int ws = (xe + 1 < nx) ? w + 1 : 0;
        T F;
        if constexpr (SPLIT) {
          const T* const left = &ed[(ws * TY + r) * 3 + k].y;
          F = ed[i].x + (ws == 0 ? peer_load(left, half ^ 1) : *left);
        } else {
          F = ed[i].x + ed[(ws * TY + r) * 3 + k].y;
        }
        if (has_src) F += (T)ssrc[(sc * 3 * TY + k * TY + r) * xp + xe];
        facc = ::fma(F, F, facc);
        if (a.fout != nullptr) {
          const size_t o = k * rcomp + (size_t)(p - 1) * rplane + (size_t)(y0 + r) * n1 + x0 + xe;
          if (F64 && a.fout_f32) reinterpret_cast<float*>(a.fout)[o] = (float)F;
          else reinterpret_cast<T*>(a.fout)[o] = F;
        }
      }
    }
  }
  cp_async_wait_all();
  if (SPLIT) cluster_sync();  // the other block may still read this one's sums
  if (timed_out) a.st->done = DONE_TIMEOUT;
  if (!FORCE) return;
  double wsum;
  if constexpr (SUMS) {
    wsum = sums.warp_total(xact, nthr);
    __syncthreads();  // the block sums use the same memory
  } else {
    double acc[8];
#pragma unroll
    for (int i = 0; i < 6; ++i) acc[i] = xact ? (0.5 / (double)kTabScale<T>) * (double)sacc[i] : 0.0;
    acc[6] = (double)facc;
    acc[7] = 0.0;
    wsum = warp_sum8(acc);
  }
  double* const red = reinterpret_cast<double*>(smraw + lay.red);
  if (a.defer) publish_partials(wsum, a.partials, red);
  else reduce_and_finalize(wsum, a.partials, a.st, a.hist, red);
}

}  // namespace hs
