// Row tiles and z chunks of the real-space pass (host).
#pragma once
#include <string.h>

#include <algorithm>
#include <vector>

#include "launch.h"
#include "real.cuh"

namespace hs {

// When the last of a real-space pass's blocks ends: yt y tiles times nz z chunks, launched y tile first, on
// `slots` equal slots, greedily; a block of a full chunk takes t, one of the last chunk t_last.
inline long long greedy_end(long long yt, long long nz, long long slots, long long t, long long t_last) {
  const long long nfull = yt * (nz - 1), a = nfull / slots, r = nfull % slots;  // r slots got one block more
  long long lo = (a + (r > 0 ? 1 : 0)) * t, hi = lo + yt * t_last;
  while (lo < hi) {  // the earliest end by which the last chunk's blocks fit on top
    const long long m = (lo + hi) / 2;
    const long long cap = (slots - r) * ((m - a * t) / t_last) + (r > 0 ? r * ((m - (a + 1) * t) / t_last) : 0);
    if (cap >= yt) hi = m;
    else lo = m + 1;
  }
  return lo;
}

// z chunk and end time of an FP64 real-space pass in yt tiles (or halves of them) of ty rows.  A warp needs 64 cycles of its
// scheduler's FP64 lanes per instruction and nearly fills them by itself, so a block of w warps takes
// (layers x voxel rows, both with their recomputed one) x max(1, w / 4) alone and an SM with more warps
// than schedulers shares that rate.  While every block is resident, SM i runs blocks i, i + nsm, ...;
// otherwise blocks follow as SMs finish.  Fewer than 8 warps on an SM do not hide its barriers (12%).  The model
// gives the measured times of 32^3 to 256^3 (chunks 1 to 64, tiles of 2, 4 and 8 rows) to about 5%: 32^3 2
// rows, chunk 1 36 us (4 rows, chunk 4, which counting resident blocks alone chose: 117 us); 64^3 4 rows,
// chunk 4 129 us (8 rows, chunk 4: 204 us); 128^3 4 rows, chunk 14 702 us (8 rows: 799); 256^3 8 rows,
// chunk 27 4850 us.
inline double pick_zchunk64(int yt, int n3, int ty, int warps, int per_sm, int nsm, int zc_min, int* zc_out) {
  const long long rows = ty + 1, fixed = 2;  // start and reduction: about two voxel rows
  const int r = std::max(1, std::min(per_sm, (4 + warps - 1) / warps));  // blocks that fill an SM's schedulers
  double best = -1;
  for (int zc = zc_min; zc <= std::max(std::min(n3, 64), zc_min); ++zc) {
    const int nz = (n3 + zc - 1) / zc, last = n3 - (nz - 1) * zc;
    const long long t = (zc + 1) * rows + fixed, t_last = (last + 1) * rows + fixed;
    const long long nblk = (long long)yt * nz, nfull = (long long)yt * (nz - 1);
    double end;
    int resident;
    if (nblk <= (long long)per_sm * nsm) {
      resident = (int)((nblk + nsm - 1) / nsm);
      long long sum = 0;
      for (int k = 0; k < resident; ++k) sum += (long long)k * nsm < nfull ? t : t_last;
      end = std::max((double)(nfull > 0 ? t : t_last), 0.25 * warps * (double)sum);
      resident = (int)std::max(1LL, nblk / nsm);
    } else {
      resident = per_sm;
      end = std::max(1.0, 0.25 * r * warps) * (double)greedy_end(yt, nz, (long long)nsm * r, t, t_last);
    }
    if (resident * warps < 8) end *= 1.12;
    if (best < 0 || end <= best) {  // the longer chunk on ties: fewer recomputed layers
      best = end;
      *zc_out = zc;
    }
  }
  return best;
}

// Planes whose sums a thread of the FP32 real-space pass keeps in FP32 registers before they go to its
// two-float sums: those of a chunk if the pass had about 1024 blocks, at most 4 (16 stress values per chain).
// Small grids, whose sums have few terms, keep chains of one plane; their passes wait for latency, not for instructions.
inline int sum_planes(int yt, int n3) {
  const int nz = std::min(n3, (1024 + yt - 1) / yt);
  return std::min(4, (n3 + nz - 1) / nz);
}

// z chunk of the FP32 real-space pass.  With w warps on an SM a plane of a block takes about 1.15 + 0.1 w
// (latency, then issue slots), so a chunk costs that for its planes, the recomputed one and a start worth
// 1.3 more, for every full wave of the resident blocks and for what is left over.  Measured at 128^3 (us): chunks
// 4 / 5 / 8 / 10 / 13 / 16 / 32: 41.9 / 38.4 / 44.2 / 34.7 / 41.3 / 41.4 / 63.7, at 256^3 16 / 24 / 26 / 29 / 32:
// 177 / 187 / 192 / 176 / 192, at 512^3 26 / 37 / 43 / 52 / 64: 1284 / 1255 / 1313 / 1281 / 1247; the model takes
// 10, 29 and 40 (1248).  The shortest chunk within 1% of the best: the tail of the last wave is the shortest too.
inline int pick_zchunk32(int yt, int n3, int warps, int per_sm, int nsm) {
  std::vector<double> cost(std::min(n3, 64) + 1, 0.0);
  double best = 1e300;
  for (int zc = 1; zc < (int)cost.size(); ++zc) {
    const long long nblk = (long long)yt * ((n3 + zc - 1) / zc), slots = (long long)per_sm * nsm;
    const long long full = nblk / slots, rem = nblk % slots;
    auto t = [&](long long b) { return 1.15 + 0.1 * (double)(b * warps); };
    cost[zc] = (zc + 2.3) * ((double)full * t(per_sm) + (rem > 0 ? t((rem + nsm - 1) / nsm) : 0.0));
    best = std::min(best, cost[zc]);
  }
  for (int zc = 1; zc < (int)cost.size(); ++zc)
    if (cost[zc] <= 1.01 * best) return zc;
  return 1;
}

// resident blocks per SM of the real-space force pass (0 if it does not run)
template <typename T> int real_occupancy(bool iso, int n1, int ty, size_t smem) {
  MarchArgs<T> a;
  memset(&a, 0, sizeof(a));
  a.n1 = n1;
  int n = 0;
  if (launch_real<T>(a, iso, ty, MODE_FORCE, dim3(1), real_threads(sizeof(T) == 8, ty, n1), smem, nullptr, &n) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// Shared memory of the real-space force pass.
inline size_t real_bytes(bool f64, int n1, int ty, bool has_src) {
  return real_layout(real_pitch(f64, ty, MODE_FORCE, n1), real_threads(f64, ty, n1), ty, has_src, f64 ? 8 : 4).total;
}

// Row tile (8, 4 or 2 rows dividing n2, its planes within smem_limit; fixed_ty > 0: this one) and z chunk of
// an FP64 real-space pass with the earliest modelled end.  Tiles of 8 rows need 255 registers, so rows of
// more than 256 columns run them in two halves (split_ok and real_rows_fit).  max_blocks > 0: at most this many blocks.
inline void pick_tile64(bool iso, int n1, int n2, int n3, int fixed_ty, size_t smem_limit, int nsm, int max_blocks,
                        bool split_ok, int* ty_out, int* zc_out) {
  *ty_out = 2;
  *zc_out = std::min(n3, 16);
  double best = -1;
  for (int ty : {8, 4, 2}) {
    if (n2 % ty != 0 || (fixed_ty > 0 && ty != fixed_ty)) continue;
    if (real_split(true, ty, n1) && !(split_ok && real_rows_fit(true, ty, n1))) continue;
    const size_t smem = real_bytes(true, n1, ty, false);
    if (smem > smem_limit) continue;
    const int occ = real_occupancy<double>(iso, n1, ty, smem);
    int zc = 0, zc_min = 1;
    const int yt = n2 / ty * real_halves(true, ty, n1);
    if (max_blocks > 0) zc_min = std::max(1, (int)(((long long)n3 * yt + max_blocks - yt) / std::max(1, max_blocks - yt)));
    const double end = pick_zchunk64(yt, n3, ty, real_threads(true, ty, n1) / 32, std::max(1, occ), nsm, std::min(zc_min, n3), &zc);
    if (best < 0 || end < best) {
      best = end;
      *ty_out = ty;
      *zc_out = zc;
    }
  }
}

}  // namespace hs
