// Three-centre recursions with one lane per shell triple (spherical basis).
//
// What bounds the 3-centre kernels on GB300 is the count of FP64 warp
// instructions: one holds its SM sub-partition's FP64 pipe for 64 clocks however
// few lanes are active.  Here every lane evaluates its own shell triple, 32
// triples of one class in lockstep, so every FP64 instruction has 32 useful
// lanes, and index arithmetic, loads and spills run in the ~60 issue slots that
// each FP64 instruction leaves free.
//
// The chain of one primitive triple (a b|c), la >= lb:
//   F_lc .. F_{lc+E}, E the bra's total angular momentum
//   -> [e|0]^(lc), e <= E: Obara-Saika over F_lc.. (registers, unrolled on E)
//   -> [e|c]^(0): lc ket steps (below), the Cartesian ket components visited
//      depth first, so three rows of e are live whatever lc is
//   -> [e|l m]: each component added into the rows of its solid harmonics
//   -> per m: bra horizontal recurrence, bra transform (or contraction with Y).
//
// Ket steps.  For a solid harmonic S_lm, S_lm(r_C) exp(-g r_C^2) is
// (2g)^-l S_lm(d/dC) exp(-g r_C^2) (Hobson's theorem), so the ket's recursion
// may drop every term that a derivative of S_lm's argument would leave as a
// factor r^2: its trace vanishes (Ahlrichs, Phys. Chem. Chem. Phys. 8 (2006)
// 3072).  What remains has two terms and lowers m by one per step,
//   [e|c+1_i]^(m) = (W-C)_i [e|c]^(m+1) + e_i/(2(p+g)) [e-1_i|c]^(m+1),
// so the bra recursion is needed at m >= lc only, and every factor is at most
// |W-C| or below one: no amplification for compact bras against diffuse kets.
// Cartesian auxiliary shells with l >= 2 hold non-harmonic parts and keep the
// general recursion (os_hgp.cuh).
#pragma once
#include "integrals.cuh"
#include "os_hgp.cuh"

namespace rihf {

// Function of a lane inside the recursion arrays: component (l, a, b) of a
// Cartesian shell l, exponents (l - a, a - b, b), 0 <= b <= a <= l.
__host__ __device__ constexpr int eidx(int l, int a, int b) { return cart_offset(l) + a * (a + 1) / 2 + b; }
// (the same from the exponents)
__host__ __device__ constexpr int ecart(int lx, int ly, int lz) {
  return cart_offset(lx + ly + lz) + (ly + lz) * (ly + lz + 1) / 2 + lz;
}
__host__ __device__ constexpr int kcart(int lx, int ly, int lz) { return (ly + lz) * (ly + lz + 1) / 2 + lz; }

// One Cartesian component of the ket's solid harmonics: function m gets coef
// times it; `first` marks a function's first component in visiting order.
struct KetTerm {
  double coef;
  int m;
  int first;
};
constexpr int kKetMaxTerms = 64;
// Terms of one auxiliary l in visiting order (cx, then cy ascending, cz the
// rest); start[v] .. start[v + 1] are those of the v-th component.
struct KetTable {
  KetTerm term[kKetMaxTerms];
  int start[ncart(kMaxLAux) + 1];
};

// Tasks of one warp claim: `n` consecutive tasks of one class.
struct LaneChunk {
  long long task0;
  int n;
  int cls;   // la | lb << 4 | lc << 8
};

// Everything a launch needs to know about one geometry.
struct LaneGeom {
  DevShells prim, aux;
  const ShellPair* pairs;
  PairTable ptab;
  const int2* tasks;
  const LaneChunk* chunks;
  const KetTable* ket;   // per auxiliary l
  double* out;           // T (integrals) or the per-atom gradient
  const double* Y;
};

// ------------------------------------------------------------ Boys function

// F[i] = F_{m0 + i}(T), i = 0..E: below the table's end one Taylor step for each
// from the nearest grid point, the weights (-d)^j / j! shared; above, the closed
// form of F_0 and upward recursion.
template <int E>
__device__ __forceinline__ void lane_boys(int m0, double T, const double* __restrict__ tab, double (&F)[E + 1]) {
  if (T < kBoysTmax) {
    const int k = __double2int_rn(T * (1.0 / kBoysStep));
    const double d = k * kBoysStep - T;
    const double* row = tab + (size_t)k * kBoysM + m0;
    double f[E + kBoysTaylor];
#pragma unroll
    for (int i = 0; i < E + kBoysTaylor; ++i) f[i] = __ldg(row + i);
    const double d2 = d * 0.5, d3 = d * (1.0 / 3.0), d4 = d * 0.25, d5 = d * 0.2, d6 = d * (1.0 / 6.0);
#pragma unroll
    for (int i = 0; i <= E; ++i) {
      double s = fma(d6, f[i + 6], f[i + 5]);
      s = fma(d5, s, f[i + 4]);
      s = fma(d4, s, f[i + 3]);
      s = fma(d3, s, f[i + 2]);
      s = fma(d2, s, f[i + 1]);
      F[i] = fma(d, s, f[i]);
    }
    return;
  }
  const double r = rsqrt(T);
  double f = 0.88622692545275801365 * r;   // sqrt(pi) / 2
  const double inv2t = 0.5 * r * r;
  // exp(-T) over F_11(T), the largest m here, is below 2^-53 from T = 72 on
  const double e = T < 72.0 ? exp(-T) : 0.0;
  for (int n = 0; n < m0; ++n) f = ((2 * n + 1) * f - e) * inv2t;
  F[0] = f;
#pragma unroll
  for (int i = 0; i < E; ++i) F[i + 1] = ((2 * (m0 + i) + 1) * F[i] - e) * inv2t;
}
static_assert(kBoysTaylor == 7, "lane_boys unrolls a seven-term Taylor step");

// ------------------------------------------------------------ bra recursion

// row[e] = [e|0]^(m0), e = 0..E, from F[i] = F_{m0 + i} times pref.
template <int E>
__device__ __forceinline__ void lane_vrr(const double (&F)[E + 1], double pref, const double (&PA)[3],
                                         const double (&WP)[3], double inv2p, double rp,
                                         double (&row)[cart_offset(E + 1)]) {
  // levels l - 2, l - 1, l over m = 0 .. E - l; the m = 0 slice is the row
  double lv[3][E + 1][ncart(E)];
#pragma unroll
  for (int m = 0; m <= E; ++m) lv[0][m][0] = pref * F[m];
  row[0] = lv[0][0][0];
  const double h[3] = {PA[0], PA[1], PA[2]};
#pragma unroll
  for (int l = 1; l <= E; ++l) {
#pragma unroll
    for (int a = 0; a <= l; ++a) {
#pragma unroll
      for (int b = 0; b <= a; ++b) {
        const int lx = l - a, ly = a - b, lz = b;
        const int i = lx > 0 ? 0 : (ly > 0 ? 1 : 2);
        const int px = lx - (i == 0), py = ly - (i == 1), pz = lz - (i == 2);
        const int n = i == 0 ? px : (i == 1 ? py : pz);   // exponent after the step down
        const int k1 = kcart(px, py, pz);
        const int k2 = n > 0 ? kcart(px - (i == 0), py - (i == 1), pz - (i == 2)) : 0;
#pragma unroll
        for (int m = 0; m <= E - l; ++m) {
          double v = h[i] * lv[(l - 1) % 3][m][k1];
          v = fma(WP[i], lv[(l - 1) % 3][m + 1][k1], v);
          if (n > 0) v = fma(n * inv2p, fma(-rp, lv[(l - 2) % 3][m + 1][k2], lv[(l - 2) % 3][m][k2]), v);
          lv[l % 3][m][kcart(lx, ly, lz)] = v;
        }
        row[eidx(l, a, b)] = lv[l % 3][0][kcart(lx, ly, lz)];
      }
    }
  }
}

// ------------------------------------------------------------ ket steps

// row[e] <- X row[e] + e_I h row[e - 1_I] for the levels e >= lo, in place (the
// higher levels first).
template <int E, int I>
__device__ __forceinline__ void lane_ket_step(double (&row)[cart_offset(E + 1)], double X, double h, int lo) {
  double eh[E + 1];
#pragma unroll
  for (int n = 1; n <= E; ++n) eh[n] = n == 1 ? h : n * h;
#pragma unroll
  for (int l = E; l >= 0; --l) {
    if (l < lo) continue;
#pragma unroll
    for (int a = 0; a <= l; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b) {
        const int lx = l - a, ly = a - b, lz = b;
        const int n = I == 0 ? lx : (I == 1 ? ly : lz);
        double v = X * row[eidx(l, a, b)];
        if (n > 0) v = fma(eh[n], row[ecart(lx - (I == 0), ly - (I == 1), lz - (I == 2))], v);
        row[eidx(l, a, b)] = v;
      }
  }
}

// Adds the primitive triple's [e|l m], EMIN <= e <= E, into K[m][e - EMIN]
// (`init`: the first triple writes).  row: [e|0]^(lc) on entry.
template <int E, int EMIN>
__device__ __forceinline__ void lane_ket(double (&row)[cart_offset(E + 1)], const double (&WQ)[3], double h, int lc,
                                         const KetTable* __restrict__ tab, bool init, double* K) {
  constexpr int O = cart_offset(EMIN), NK = cart_offset(E + 1) - O;
  auto emit = [&](const double (&z)[cart_offset(E + 1)], int v) {
    const int t1 = tab->start[v + 1];
#pragma unroll 1
    for (int t = tab->start[v]; t < t1; ++t) {
      const KetTerm q = tab->term[t];
      double* k = K + q.m * NK;
      if (q.first && init) {
        if (q.coef == 1.0) {
#pragma unroll
          for (int e = 0; e < NK; ++e) k[e] = z[O + e];
        } else {
#pragma unroll
          for (int e = 0; e < NK; ++e) k[e] = q.coef * z[O + e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < NK; ++e) k[e] = fma(q.coef, z[O + e], k[e]);
      }
    }
  };
  if (lc == 0) {
    emit(row, 0);
    return;
  }
  double y[cart_offset(E + 1)], z[cart_offset(E + 1)];
  int v = 0;
#pragma unroll 1
  for (int cx = 0; cx <= lc; ++cx) {
#pragma unroll
    for (int e = 0; e < cart_offset(E + 1); ++e) y[e] = row[e];
#pragma unroll 1
    for (int cy = 0; cy <= lc - cx; ++cy) {
#pragma unroll
      for (int e = 0; e < cart_offset(E + 1); ++e) z[e] = y[e];
      // the steps left after this one may lower e by one each
#pragma unroll 1
      for (int s = cx + cy + 1; s <= lc; ++s) lane_ket_step<E, 2>(z, WQ[2], h, EMIN - (lc - s));
      emit(z, v++);
      if (cy < lc - cx) lane_ket_step<E, 1>(y, WQ[1], h, EMIN - (lc - (cx + cy + 1)));
    }
    if (cx < lc) lane_ket_step<E, 0>(row, WQ[0], h, EMIN - (lc - (cx + 1)));
  }
}

// ------------------------------------------------------------ bra HRR

// One level of (a b+1_i| = (a+1_i b| + AB_i (a b|: from rows a in [LA, LA+LB-B+1]
// of b = B - 1 to rows a in [LA, LA+LB-B] of b = B (rows offset by a = LA).
template <int LA, int TOP, int B>
__device__ __forceinline__ void lane_hrr_level(const double* prev, double* cur, const double (&AB)[3]) {
  constexpr int O = cart_offset(LA);
#pragma unroll
  for (int l = LA; l <= TOP; ++l)
#pragma unroll
    for (int a = 0; a <= l; ++a)
#pragma unroll
      for (int c = 0; c <= a; ++c)
#pragma unroll
        for (int p = 0; p <= B; ++p)
#pragma unroll
          for (int q = 0; q <= p; ++q) {
            const int ax = l - a, ay = a - c, az = c, bx = B - p, by = p - q, bz = q;
            const int i = bx > 0 ? 0 : (by > 0 ? 1 : 2);
            const int kb = kcart(bx - (i == 0), by - (i == 1), bz - (i == 2));
            const int r1 = ecart(ax + (i == 0), ay + (i == 1), az + (i == 2)) - O, r0 = ecart(ax, ay, az) - O;
            cur[(r0)*ncart(B) + kcart(bx, by, bz)] = fma(AB[i], prev[r0 * ncart(B - 1) + kb], prev[r1 * ncart(B - 1) + kb]);
          }
}

// (la lb| for one ket function from k[e - LA], e in [LA, LA + LB]:
// out[ka * ncart(LB) + kb].
template <int LA, int LB>
__device__ __forceinline__ void lane_hrr(const double* k, const double (&AB)[3], double* out) {
  if constexpr (LB == 0) {
#pragma unroll
    for (int i = 0; i < ncart(LA); ++i) out[i] = k[i];
  } else if constexpr (LB == 1) {
    lane_hrr_level<LA, LA, 1>(k, out, AB);
  } else if constexpr (LB == 2) {
    double h1[(cart_offset(LA + 2) - cart_offset(LA)) * 3];
    lane_hrr_level<LA, LA + 1, 1>(k, h1, AB);
    lane_hrr_level<LA, LA, 2>(h1, out, AB);
  } else {
    double h1[(cart_offset(LA + 3) - cart_offset(LA)) * 3], h2[(cart_offset(LA + 2) - cart_offset(LA)) * 6];
    lane_hrr_level<LA, LA + 2, 1>(k, h1, AB);
    lane_hrr_level<LA, LA + 1, 2>(h1, h2, AB);
    lane_hrr_level<LA, LA, 3>(h2, out, AB);
  }
}

// ------------------------------------------------------------ bra solid harmonics

// Coefficient of Cartesian component (x, y, z) in the real solid harmonic m of
// degree l <= 4, every function with the norm of x^l (the library's rows of the
// transform table, spelt out so that the zeros cost nothing).
__host__ __device__ constexpr double bra_sph(int l, int m, int x, int y, int z) {
  if (l == 0) return 1.0;
  if (l == 1) return (m == -1 && y) || (m == 0 && z) || (m == 1 && x) ? 1.0 : 0.0;
  constexpr double s3 = 1.7320508075688772935, s15 = 3.8729833462074168852;
  constexpr double s58 = 0.79056941504209483300, s38 = 0.61237243569579452455;
  if (l == 2) {
    if (m == -2) return x == 1 && y == 1 ? s3 : 0.0;
    if (m == -1) return y == 1 && z == 1 ? s3 : 0.0;
    if (m == 0) return z == 2 ? 1.0 : (x == 2 || y == 2 ? -0.5 : 0.0);
    if (m == 1) return x == 1 && z == 1 ? s3 : 0.0;
    return x == 2 ? 0.5 * s3 : (y == 2 ? -0.5 * s3 : 0.0);
  }
  if (l == 4) {
    constexpr double s5 = 2.2360679774997896964, s35 = 5.9160797830996160426, s70 = 8.3666002653407554798;
    if (m == -4) return x == 3 && y == 1 ? 0.5 * s35 : (x == 1 && y == 3 ? -0.5 * s35 : 0.0);
    if (m == -3) return z == 1 && x == 2 ? 0.75 * s70 : (z == 1 && y == 3 ? -0.25 * s70 : 0.0);
    if (m == -2) return x == 1 && y == 1 ? 3.0 * s5 : ((x == 3 && y == 1) || (x == 1 && y == 3) ? -0.5 * s5 : 0.0);
    if (m == -1) return y == 1 && z == 3 ? 4.0 * s58 : (z == 1 && (y == 3 || (x == 2 && y == 1)) ? -3.0 * s58 : 0.0);
    if (m == 0)
      return z == 4 ? 1.0 : (z == 2 ? (x == 2 || y == 2 ? -3.0 : 0.0) : (z == 0 ? (x == 2 ? 0.75 : (x == 4 || y == 4 ? 0.375 : 0.0)) : 0.0));
    if (m == 1) return x == 1 && z == 3 ? 4.0 * s58 : (z == 1 && (x == 3 || (x == 1 && y == 2)) ? -3.0 * s58 : 0.0);
    if (m == 2)
      return z == 2 ? (x == 2 ? 1.5 * s5 : (y == 2 ? -1.5 * s5 : 0.0)) : (x == 4 ? -0.25 * s5 : (y == 4 ? 0.25 * s5 : 0.0));
    if (m == 3) return z == 1 && x == 3 ? 0.25 * s70 : (z == 1 && x == 1 && y == 2 ? -0.75 * s70 : 0.0);
    return x == 4 || y == 4 ? 0.125 * s35 : (x == 2 && y == 2 ? -0.75 * s35 : 0.0);
  }
  if (m == -3) return x == 2 && y == 1 ? 3.0 * s58 : (y == 3 ? -s58 : 0.0);
  if (m == -2) return x == 1 && y == 1 && z == 1 ? s15 : 0.0;
  if (m == -1) return y == 1 && z == 2 ? 4.0 * s38 : ((x == 2 && y == 1) || y == 3 ? -s38 : 0.0);
  if (m == 0) return z == 3 ? 1.0 : (z == 1 && (x == 2 || y == 2) ? -1.5 : 0.0);
  if (m == 1) return x == 1 && z == 2 ? 4.0 * s38 : (x == 3 || (x == 1 && y == 2) ? -s38 : 0.0);
  if (m == 2) return z == 1 && x == 2 ? 0.5 * s15 : (z == 1 && y == 2 ? -0.5 * s15 : 0.0);
  return x == 3 ? s58 : (x == 1 && y == 2 ? -3.0 * s58 : 0.0);
}

// Sum over the components of one shell: dst[m] (stride SD) = sum_k coef src[k]
// (stride SS), FWD; or dst[k] = sum_m coef src[m], transposed.
template <int L, bool FWD>
__device__ __forceinline__ void lane_sph(const double* src, int ss, double* dst, int sd) {
  if constexpr (L == 0) {
    dst[0] = src[0];
  } else if constexpr (FWD) {
#pragma unroll
    for (int m = -L; m <= L; ++m) {
      double v = 0.0;
      bool has = false;
#pragma unroll
      for (int a = 0; a <= L; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          const double c = bra_sph(L, m, L - a, a - b, b);
          if (c != 0.0) {
            const double s = src[kcart(L - a, a - b, b) * ss];
            v = has ? fma(c, s, v) : (c == 1.0 ? s : c * s);
            has = true;
          }
        }
      dst[(m + L) * sd] = v;
    }
  } else {
#pragma unroll
    for (int a = 0; a <= L; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b) {
        double v = 0.0;
        bool has = false;
#pragma unroll
        for (int m = -L; m <= L; ++m) {
          const double c = bra_sph(L, m, L - a, a - b, b);
          if (c != 0.0) {
            const double s = src[(m + L) * ss];
            v = has ? fma(c, s, v) : (c == 1.0 ? s : c * s);
            has = true;
          }
        }
        dst[kcart(L - a, a - b, b) * sd] = v;
      }
  }
}

// ------------------------------------------------------------ one primitive triple

// [e|l m] of the pair primitive q and the auxiliary primitive ic of shell centre
// C, added into K (written when init).
template <int E, int EMIN>
__device__ __forceinline__ void lane_triple(const PairPrim& q, const DevShells& aux, int ic, const double (&C)[3], int lc,
                                            const double* __restrict__ boys, const KetTable* __restrict__ tab,
                                            bool init, double* K) {
  const double g = aux.exps[ic], ig = aux.iexps[ic], cc = aux.coefs[ic];
  const double CP[3] = {C[0] - q.P[0], C[1] - q.P[1], C[2] - q.P[2]};
  const double R2 = fma(CP[0], CP[0], fma(CP[1], CP[1], CP[2] * CP[2]));
  const double r = rsqrt(q.p + g);          // (p + g)^{-1/2}
  const double ipq = r * r;
  const double gi = g * ipq, pi = q.p * ipq;
  const double WP[3] = {gi * CP[0], gi * CP[1], gi * CP[2]};
  const double WQ[3] = {-pi * CP[0], -pi * CP[1], -pi * CP[2]};
  double F[E + 1];
  lane_boys<E>(lc, q.p * gi * R2, boys, F);
  double row[cart_offset(E + 1)];
  lane_vrr<E>(F, q.K * (cc * ig) * r, q.PA, WP, 0.5 * q.inv_p, gi, row);
  lane_ket<E, EMIN>(row, WQ, 0.5 * ipq, lc, tab, init, K);
}

// ------------------------------------------------------------ work claims

// The next chunk of the launch for this warp; false when none is left.  One
// geometry (ngeom 0): G0's list; a batch: chunk c belongs to the geometry g with
// off[g] <= c < off[g + 1].
__device__ __forceinline__ bool lane_claim(const LaneGeom& G0, const LaneGeom* __restrict__ geoms,
                                           const long long* __restrict__ off, int ngeom, long long nchunk, int* counter,
                                           const LaneGeom*& G, LaneChunk& ch) {
  int t = 0;
  if ((threadIdx.x & 31) == 0) t = atomicAdd(counter, 1);
  t = __shfl_sync(0xffffffffu, t, 0);
  if (t >= nchunk) return false;
  if (ngeom == 0) {
    G = &G0;
    ch = G0.chunks[t];
    return true;
  }
  int lo = 0, hi = ngeom;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= t) lo = mid;
    else hi = mid;
  }
  G = geoms + lo;
  ch = G->chunks[t - off[lo]];
  return true;
}

// Index of (row, col), any order, in a pair-packed slice.
__device__ __forceinline__ long long lane_tri(long long i, long long j) {
  return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i;
}

}  // namespace rihf

namespace rihf {

// Class groups of a launch: la + lb <= 2 (ss, ps, pp, ds); (d p, d d; f shells.
constexpr int kLaneGroups = 3;
__host__ __device__ constexpr int lane_group(int la, int lb) { return la >= 3 ? 2 : (la + lb <= 2 ? 0 : 1); }
// Resident one-warp blocks per SM of the two kernels, by group.
constexpr int kLaneBlocks[kLaneGroups] = {12, 8, 8};

// Runs f<la, lb>() for the pair class of cls, a class of group GRP.
#define RIHF_LANE_CASE(a, b) \
  case (a) | (b) << 4: f.template run<a, b>(); break;
template <int GRP, class F>
__device__ __forceinline__ void lane_dispatch(int cls, F f) {
  if constexpr (GRP == 0) {
    switch (cls & 0xff) {
      RIHF_LANE_CASE(0, 0)
      RIHF_LANE_CASE(1, 0)
      RIHF_LANE_CASE(1, 1)
      RIHF_LANE_CASE(2, 0)
    }
  } else if constexpr (GRP == 1) {
    switch (cls & 0xff) {
      RIHF_LANE_CASE(2, 1)
      RIHF_LANE_CASE(2, 2)
    }
  } else {
    switch (cls & 0xff) {
      RIHF_LANE_CASE(3, 0)
      RIHF_LANE_CASE(3, 1)
      RIHF_LANE_CASE(3, 2)
      RIHF_LANE_CASE(3, 3)
    }
  }
}
#undef RIHF_LANE_CASE

// One geometry's lane tasks: chunk lists by group (device) and their lengths.
struct LaneTasks {
  LaneGeom geom{};                       // chunks unset
  const LaneChunk* chunks[kLaneGroups] = {};
  long long nchunk[kLaneGroups] = {};
};

// Host side: the tasks of every (pair, auxiliary shell), class by class, inside
// a class atom triple by atom triple (a lane's consecutive tasks then mostly
// share their atoms, so the derivative kernel flushes its sums rarely), and the
// chunks that the warps claim, heaviest class first.
void build_lane_tasks(const std::vector<ShellPair>& pairs, const std::vector<int>& lprim, const std::vector<int>& patom,
                      const std::vector<int>& laux, const std::vector<int>& aatom, int sms, std::vector<int2>& tasks,
                      std::vector<LaneChunk> (&chunks)[kLaneGroups]);
// The ket tables of every auxiliary l from the transform table (kTrL x
// kTrStride x kTrStride, rows: functions).
std::vector<KetTable> build_ket_tables(const std::vector<double>& tr, const std::vector<int>& nf);

// FP64 operations (an FMA counts two) of the two kernels over every task, from
// the loops of their recursions.
void lane_flops(const std::vector<ShellPair>& pairs, const std::vector<int>& lprim, const std::vector<int>& nprim,
                const std::vector<int>& patom, const std::vector<int>& laux, const std::vector<int>& naux_prim,
                const std::vector<int>& aatom, const std::vector<KetTable>& ket, double* eri3, double* grad3);

// Device tables of a batched launch: per group the geometries' descriptors and
// chunk offsets.
struct LaneBatchTables {
  LaneGeom* geoms = nullptr;   // kLaneGroups x cap
  long long* off = nullptr;    // kLaneGroups x (cap + 1)
  int cap = 0;
};
// (mu nu|P) of one geometry into its geom.out, or of a batch.
void launch_lane_eri3(const IntegralCtx& ic, int sms, const LaneTasks& t);
void launch_lane_eri3_batch(const IntegralCtx& ic, int sms, const std::vector<LaneTasks>& batch, LaneBatchTables& t);
// The derivative contraction of one geometry with geom.Y, added into geom.out
// (per atom), or of a batch.
void launch_lane_grad(const IntegralCtx& ic, int sms, const LaneTasks& t);
void launch_lane_grad_batch(const IntegralCtx& ic, int sms, const std::vector<LaneTasks>& batch, LaneBatchTables& t);

// Host side shared by the two batched launches: group g's descriptors and
// offsets into t (copied on ic.stream and waited for); the chunk count.
long long lane_batch_tables(const IntegralCtx& ic, const std::vector<LaneTasks>& batch, int g, LaneBatchTables& t);

}  // namespace rihf
