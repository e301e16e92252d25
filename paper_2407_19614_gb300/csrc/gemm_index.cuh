// Launch plan and index arithmetic of the FP64 GEMM (linalg.cu), kept apart from the
// kernel so that a host program can walk every address that a launch forms.
#pragma once
#include <algorithm>
#include <cmath>

#include "../../include/rihf.h"
#include "linalg.cuh"

namespace rihf {

// C tiles of 16 x 16 by 128-thread CTAs, two elements a thread.  FP64 bounds every
// product here (two FMAs per clock and SM), so what counts is that no tile is
// mostly padding and that the tiles fill the SMs evenly: 16 is the largest tile
// that gives a 192 x 192 result one CTA per SM (144) without splitting K, and wastes
// least at the 40 columns of H = B C~ (48 computed; 64 with a 32-wide tile).  The
// operands come through a ring of three K chunks filled by cp.async two chunks
// ahead.  Measured, 192 x 192 x 192: 18 us, 14 us for a symmetric result, against
// 17 us plus a 5 us reduction of split sums with 32 x 32 tiles; H and K of an FP64
// Fock build at N = 192, Naux = 848 (40 occupied): 3.6 ms against 5.7.
constexpr int GT = 16;        // output tile
constexpr int GK = 32;        // K chunk, at most
constexpr int GS = 3;         // chunks in flight
constexpr int GThreads = 128;
constexpr int kGemmCluster = 8;   // most K slices summed through a thread-block cluster

// What a launch covers: grid (ctas, nslice).
struct GemmPlan {
  long long ctas = 0;              // tiles x batches
  int tiles = 0, tn = 0;           // tiles of a result, tile columns
  int nslice = 1, kper = 0, bper = 0;
  int chunk = 1, cluster = 0;
};

inline GemmPlan gemm_plan(const GemmArgs& g, int sms, size_t work_elems) {
  GemmPlan p;
  const int tm = ceil_div(g.M, GT);
  p.tn = ceil_div(g.N, GT);
  const int nb = g.reduce_batch ? 1 : g.batch;
  if ((long long)tm * p.tn > 0x7fffffffLL / nb)
    throw RihfError(RIHF_ERR_INVALID_ARG, "dgemm: too many tiles for this product shape");
  p.tiles = g.lower_only ? tm * (tm + 1) / 2 : tm * p.tn;
  // the chunk divides K when K is short (reduced batches of K = nocc: no padded steps)
  p.chunk = std::max(1, ceil_div(g.K, ceil_div(std::max(1, g.K), GK)));
  // Slices: the least time of the fullest SM, in FP64 steps of one tile: a CTA alone
  // on its SM takes 1.75 times its FP64 time (one warp per sub-partition: 226 clocks
  // a step instead of 128, measured at 192 x 192 x 192), so two half slices beat one
  // whole; and a slice costs some steps beside its own (filling the ring, the sum).
  // Up to kGemmCluster slices are summed in a cluster; more go through the workspace,
  // which has to hold them, and only where a long reduction leaves each slice long.
  p.ctas = (long long)p.tiles * nb;
  const long long len = g.reduce_batch ? (long long)g.batch * g.K : g.K;
  const long long most_len = g.reduce_batch ? g.batch : std::max(1, g.K / 8);   // at least 8 of K a slice
  double best = 1e300;
  for (int s = 1; s <= 64 && s <= most_len; ++s) {
    if (s > kGemmCluster &&
        ((size_t)s * g.M * g.N * nb > work_elems || len / s < 512)) break;
    const double steps = (double)ceil_div(len, s) + (s > 1 ? 16.0 : 8.0) + (s > kGemmCluster ? 40.0 : 0.0);
    const double cost = std::max((double)((p.ctas * s + sms - 1) / sms), 1.75) * steps;
    if (cost < 0.98 * best) {
      best = cost;
      p.nslice = s;
    }
  }
  p.kper = g.K;
  p.bper = g.batch;
  if (g.reduce_batch) {
    p.bper = ceil_div(g.batch, p.nslice);
    p.nslice = ceil_div(g.batch, p.bper);
  } else if (p.nslice > 1) {
    p.kper = ceil_div(g.K, p.nslice);
    p.nslice = ceil_div(g.K, p.kper);
  }
  p.cluster = p.nslice > 1 && p.nslice <= kGemmCluster ? 1 : 0;
  return p;
}

// Tile t of the result: all tiles row by row, or (lower_only) those on and below
// the diagonal.
__host__ __device__ __forceinline__ void gemm_tile(const GemmArgs& g, int t, int tn, int& tm, int& tc) {
  if (!g.lower_only) {
    tm = t / tn;
    tc = t - tm * tn;
    return;
  }
  tm = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while (tm * (tm + 1) / 2 > t) --tm;
  while ((tm + 1) * (tm + 2) / 2 <= t) ++tm;
  tc = t - tm * (tm + 1) / 2;
}

// Share of block (bx, by): its tile's origin, the batches [b0, b1) and the k range
// [k0, k1) that it sums, in `total` chunks, `per` of them a batch.
struct GemmBlock {
  int batch, m0, n0, b0, b1, k0, k1, per, total;
};
__host__ __device__ __forceinline__ GemmBlock gemm_block(const GemmArgs& g, int bx, int by, int tiles, int tn, int kper,
                                                         int bper, int chunk) {
  GemmBlock q;
  q.batch = bx / tiles;
  int tm, tc;
  gemm_tile(g, bx - q.batch * tiles, tn, tm, tc);
  q.m0 = tm * GT;
  q.n0 = tc * GT;
  q.b0 = q.batch;
  q.b1 = q.batch + 1;
  q.k0 = 0;
  q.k1 = g.K;
  if (g.reduce_batch) {
    q.b0 = by * bper;
    q.b1 = g.batch < q.b0 + bper ? g.batch : q.b0 + bper;
  } else {
    q.k0 = by * kper;
    q.k1 = g.K < q.k0 + kper ? g.K : q.k0 + kper;
  }
  q.per = q.k1 > q.k0 ? (q.k1 - q.k0 + chunk - 1) / chunk : 0;
  q.total = q.b1 > q.b0 ? (q.b1 - q.b0) * q.per : 0;
  return q;
}

// Copy number idx (0 .. GT * chunk - 1) of one operand's chunk at kc: row and k in the
// tile, and the source's offset (0, not to be read, for elements that do not exist).
// KFAST: k is the contiguous index.
struct GemmElem {
  int row, k;
  bool valid;
  long long at;
};
template <bool KFAST>
__host__ __device__ __forceinline__ GemmElem gemm_elem(int idx, int chunk, int row0, int rows, int kc, int k1, int ld) {
  GemmElem e;
  if (KFAST) {
    e.k = idx % chunk;
    e.row = idx / chunk;
  } else {
    e.row = idx % GT;
    e.k = idx / GT;
  }
  const int r = row0 + e.row, x = kc + e.k;
  e.valid = r < rows && x < k1;
  e.at = !e.valid ? 0 : KFAST ? (long long)r * ld + x : (long long)x * ld + r;
  return e;
}

}  // namespace rihf
