// Contraction of lane-held integrals with a Cartesian weight block Y: the sums
// that the derivative kernels need (see grad_eri3_lane.cu).
#pragma once
#include "eri3_lane.cuh"

namespace rihf {

// w of the level b = B - 1 over a in [LA, TOP + 1] from the level b = B over
// a in [LA, TOP]: the transpose of lane_hrr_level.
template <int LA, int TOP, int B>
__device__ __forceinline__ void lane_hrr_adjoint(const double* hi, double* lo, const double (&AB)[3]) {
  constexpr int O = cart_offset(LA);
#pragma unroll
  for (int l = LA; l <= TOP + 1; ++l)
#pragma unroll
    for (int a = 0; a <= l; ++a)
#pragma unroll
      for (int c = 0; c <= a; ++c)
#pragma unroll
        for (int p = 0; p <= B - 1; ++p)
#pragma unroll
          for (int q = 0; q <= p; ++q) {
            const int ax = l - a, ay = a - c, az = c, bx = B - 1 - p, by = p - q, bz = q;
            double v = 0.0;
            bool has = false;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              // (b + 1_i) is built along direction i when i is its first one
              const bool mine = i == 0 || (i == 1 && bx == 0) || (i == 2 && bx == 0 && by == 0);
              if (!mine) continue;
              const int kb = kcart(bx + (i == 0), by + (i == 1), bz + (i == 2));
              const int ai = i == 0 ? ax : (i == 1 ? ay : az);
              if (l > LA && ai > 0) {
                const double s = hi[(ecart(ax - (i == 0), ay - (i == 1), az - (i == 2)) - O) * ncart(B) + kb];
                v = has ? v + s : s;
                has = true;
              }
              if (l <= TOP) {
                const double s = hi[(ecart(ax, ay, az) - O) * ncart(B) + kb];
                v = has ? fma(AB[i], s, v) : AB[i] * s;
                has = true;
              }
            }
            lo[(ecart(ax, ay, az) - O) * ncart(B - 1) + kcart(bx, by, bz)] = v;
          }
}

// w[e - LA], e in [LA, LA + LB], from Ycart[ka * ncart(LB) + kb].
template <int LA, int LB>
__device__ __forceinline__ void lane_weights(const double* y, const double (&AB)[3], double* w) {
  if constexpr (LB == 0) {
#pragma unroll
    for (int i = 0; i < ncart(LA); ++i) w[i] = y[i];
  } else if constexpr (LB == 1) {
    lane_hrr_adjoint<LA, LA, 1>(y, w, AB);
  } else if constexpr (LB == 2) {
    double h1[(cart_offset(LA + 2) - cart_offset(LA)) * 3];
    lane_hrr_adjoint<LA, LA, 2>(y, h1, AB);
    lane_hrr_adjoint<LA, LA + 1, 1>(h1, w, AB);
  } else {
    double h2[(cart_offset(LA + 2) - cart_offset(LA)) * 6], h1[(cart_offset(LA + 3) - cart_offset(LA)) * 3];
    lane_hrr_adjoint<LA, LA, 3>(y, h2, AB);
    lane_hrr_adjoint<LA, LA + 1, 2>(h2, h1, AB);
    lane_hrr_adjoint<LA, LA + 2, 1>(h1, w, AB);
  }
}

// The sums of one ket function: s = {U[3], D[3], B[3], V} += ...; k[e - EMIN]
// the integrals, y the Cartesian Y block.
template <int LA, int LB>
__device__ __forceinline__ void lane_contract(const double* k, const double* y, const double (&AB)[3], double (&s)[10]) {
  constexpr int EMIN = LA > 0 ? LA - 1 : 0, OK = cart_offset(EMIN), OW = cart_offset(LA);
  if constexpr (LB > 0) {
    double q[ncart(LA) * ncart(LB - 1)];
    lane_hrr<LA, LB - 1>(k + (OW - OK), AB, q);
#pragma unroll
    for (int ka = 0; ka < ncart(LA); ++ka)
#pragma unroll
      for (int p = 0; p <= LB; ++p)
#pragma unroll
        for (int c = 0; c <= p; ++c) {
          const int b[3] = {LB - p, p - c, c};
          const double yv = y[ka * ncart(LB) + kcart(b[0], b[1], b[2])];
#pragma unroll
          for (int i = 0; i < 3; ++i)
            if (b[i] > 0) {
              const double yb = b[i] == 1 ? yv : b[i] * yv;
              s[6 + i] = fma(yb, q[ka * ncart(LB - 1) + kcart(b[0] - (i == 0), b[1] - (i == 1), b[2] - (i == 2))], s[6 + i]);
            }
        }
  }
  double w[cart_offset(LA + LB + 1) - OW];
  lane_weights<LA, LB>(y, AB, w);
#pragma unroll
  for (int l = LA; l <= LA + LB; ++l)
#pragma unroll
    for (int a = 0; a <= l; ++a)
#pragma unroll
      for (int c = 0; c <= a; ++c) {
        const int e[3] = {l - a, a - c, c};
        const double we = w[ecart(e[0], e[1], e[2]) - OW];
        s[9] = fma(we, k[ecart(e[0], e[1], e[2]) - OK], s[9]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          s[i] = fma(we, k[ecart(e[0] + (i == 0), e[1] + (i == 1), e[2] + (i == 2)) - OK], s[i]);
          if (e[i] > 0) {
            const double wi = e[i] == 1 ? we : e[i] * we;
            s[3 + i] = fma(wi, k[ecart(e[0] - (i == 0), e[1] - (i == 1), e[2] - (i == 2)) - OK], s[3 + i]);
          }
        }
      }
}

}  // namespace rihf
