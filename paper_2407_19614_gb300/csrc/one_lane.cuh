// Shared by the one-electron kernels of spherical bases (one_lane.cu,
// grad_one_lane.cu).
#pragma once
#include "grad_lane.cuh"
#include "lane2.cuh"

namespace rihf {

// Gaussian product of two primitives.
struct Prod {
  double p, ip, K;      // exponent sum, 1/p, exp(-ab/p R^2)
  double P[3], PA[3];
};
__device__ __forceinline__ Prod gauss_prod(double al, double be, const double (&A)[3], const double (&AB)[3]) {
  Prod q;
  q.p = al + be;
  q.ip = 1.0 / q.p;
  const double f = be * q.ip;
  double r2 = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q.PA[i] = -f * AB[i];
    q.P[i] = A[i] + q.PA[i];
    r2 = fma(AB[i], AB[i], r2);
  }
  q.K = exp(-al * f * r2);
  return q;
}

// s[i * ld + j], i <= I, j <= J: 1D overlaps of x_A^i and x_B^j over the Gaussian
// product, s0 = sqrt(pi / p).  PB = PA + AB.
template <int I, int J, int LD>
__device__ __forceinline__ void overlap_1d(double PA, double PB, double inv2p, double s0, double* s) {
  s[0] = s0;
#pragma unroll
  for (int i = 1; i <= I; ++i) {
    double v = PA * s[(i - 1) * LD];
    if (i >= 2) v = fma((i - 1) * inv2p, s[(i - 2) * LD], v);
    s[i * LD] = v;
  }
#pragma unroll
  for (int j = 1; j <= J; ++j)
#pragma unroll
    for (int i = 0; i <= I; ++i) {
      double v = PB * s[i * LD + j - 1];
      if (j >= 2) v = fma((j - 1) * inv2p, s[i * LD + j - 2], v);
      if (i >= 1) v = fma(i * inv2p, s[(i - 1) * LD + j - 1], v);
      s[i * LD + j] = v;
    }
}
// The kinetic partner (second derivative on b) of s[i][j].
__device__ __forceinline__ double second_1d(const double* s, int LD, int i, int j, double be) {
  double v = 4.0 * be * be * s[i * LD + j + 2] - 2.0 * be * (2 * j + 1) * s[i * LD + j];
  if (j >= 2) v += j * (j - 1) * s[i * LD + j - 2];
  return v;
}

// Cartesian (la, lb) block -> spherical.
template <int LA, int LB>
__device__ __forceinline__ void bra_block(const double* cart, double* out) {
  double half[ncart(LA) * nsph(LB)];
#pragma unroll
  for (int ka = 0; ka < ncart(LA); ++ka) lane_sph<LB, true>(cart + ka * ncart(LB), 1, half + ka * nsph(LB), 1);
#pragma unroll
  for (int b = 0; b < nsph(LB); ++b) lane_sph<LA, true>(half + b, nsph(LB), out + b, nsph(LB));
}
// Spherical block M[row0 + a][col0 + b] -> Cartesian weights.
template <int LA, int LB>
__device__ __forceinline__ void weight_block(const double* __restrict__ M, int N, int mu0, int nu0, double* y) {
  constexpr int FA = nsph(LA), FB = nsph(LB);
  double z[FA * FB], half[ncart(LA) * FB];
#pragma unroll
  for (int a = 0; a < FA; ++a)
#pragma unroll
    for (int b = 0; b < FB; ++b) z[a * FB + b] = __ldg(M + (size_t)(mu0 + a) * N + nu0 + b);
#pragma unroll
  for (int b = 0; b < FB; ++b) lane_sph<LA, false>(z + b, FB, half + b, FB);
#pragma unroll
  for (int ka = 0; ka < ncart(LA); ++ka) lane_sph<LB, false>(half + ka * FB, 1, y + ka * ncart(LB), 1);
}

struct OneArgs {
  DevShells prim;
  const int2* tasks;
  const LaneChunk* chunks;
  int lanes;      // per pair: 4, 8, 16 or 32
  int natoms;
  const int* Z;
  const double* axyz;
  const double* boys;
};

inline OneArgs one_args(const IntegralCtx& ic, const DevShells& prim, const Lane2Tasks& t, int lanes, int natoms,
                        const int* Z, const double* axyz) {
  return OneArgs{prim, t.tasks, t.chunks, lanes, natoms, Z, axyz, ic.boys};
}

// The pairs of this warp: lanes / 4 blocks a chunk, 32 / lanes pairs each (a short
// chunk's last blocks have none: false).
__device__ __forceinline__ bool one_chunk(const OneArgs& g, LaneChunk& ch) {
  const int blocks = g.lanes / (32 / kOneChunk), per = 32 / g.lanes;
  ch = g.chunks[blockIdx.x / blocks];
  const int at = (blockIdx.x % blocks) * per;
  ch.task0 += at;
  ch.n = min(per, ch.n - at);
  return ch.n > 0;
}
inline unsigned one_grid(const Lane2Tasks& t, int lanes) { return (unsigned)(t.nchunk * (lanes / (32 / kOneChunk))); }

// Runs f<la, lb>(g, ch, ...) for the class of chunk ch.
#define RIHF_ONE_CASES(f, ...)                          \
  switch (ch.cls & 0xff) {                              \
    case 0x00: f<0, 0>(g, ch, __VA_ARGS__); break;      \
    case 0x01: f<1, 0>(g, ch, __VA_ARGS__); break;      \
    case 0x11: f<1, 1>(g, ch, __VA_ARGS__); break;      \
    case 0x02: f<2, 0>(g, ch, __VA_ARGS__); break;      \
    case 0x12: f<2, 1>(g, ch, __VA_ARGS__); break;      \
    case 0x22: f<2, 2>(g, ch, __VA_ARGS__); break;      \
    case 0x03: f<3, 0>(g, ch, __VA_ARGS__); break;      \
    case 0x13: f<3, 1>(g, ch, __VA_ARGS__); break;      \
    case 0x23: f<3, 2>(g, ch, __VA_ARGS__); break;      \
    default: f<3, 3>(g, ch, __VA_ARGS__); break;        \
  }

}  // namespace rihf
