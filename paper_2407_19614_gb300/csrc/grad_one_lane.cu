// Derivative contraction of the one-electron integrals for spherical bases:
// 4 to 32 lanes per shell pair (one_lanes), which share out the nuclei and, for
// overlap and kinetic energy, the Cartesian components.
//
// The derivative of nuclear attraction needs the weights w of the horizontal
// recurrence applied to D (grad_lane.cuh) once per pair; each nucleus then costs
// its recursion and one pass of dot products, its own force being minus the
// translation 2p U - D + 2 beta AB V of the pair.  (A, B) terms are linear in the
// integrals and are contracted once, from the sum over nuclei.
// Bound by FP64 instructions, at small sizes by the latency of one pair.  0.086 ms at
// (H2O)3 (666 pairs, 9 nuclei), 0.137 at (H2O)8, 1.08 at (H2O)10 in the larger basis; the
// warp-cooperative kernel (a task per pair and nucleus, four recurrences each) takes
// 0.105, 0.95 and 16.4 ms.  One water in the larger basis is the one case where it is
// ahead, 0.182 against 0.195 ms: the serial chain of an (f f| pair.
#include <algorithm>

#include "../../include/rihf.h"
#include "one_lane.cuh"

namespace rihf {

namespace {

// The contraction out of line for the f classes: once per pair, and the compiler
// takes far longer over one large function than over two.
template <int LA, int LB>
__device__ __noinline__ void contract_call(const double* k, const double* y, const double (&AB)[3], double (&s)[10]) {
  lane_contract<LA, LB>(k, y, AB, s);
}

template <int LA, int LB>
__device__ __noinline__ void grad_one_tasks(const OneArgs& g, const LaneChunk& ch, const double* __restrict__ D,
                                            const double* __restrict__ Wm, double* grad_one, double* grad_ovl) {
  constexpr int E = LA + LB + 1, EMIN = LA > 0 ? LA - 1 : 0, O = cart_offset(EMIN), NK = cart_offset(E + 1) - O;
  constexpr int NA = ncart(LA), NB = ncart(LB), OW = cart_offset(LA), NW = cart_offset(LA + LB + 1) - OW, LD = LB + 3;
  constexpr int kUnroll = LA + LB < 6 ? 64 : 1;   // (f f|: rolled, for the compiler's sake
  const int L = g.lanes, lane = threadIdx.x, q = lane & (L - 1), slot = lane >> (31 - __clz(L));
  const int j = min(slot, ch.n - 1);
  const bool live = slot < ch.n;
  const DevShells& pr = g.prim;
  const int2 tk = g.tasks[ch.task0 + j];
  const int sa = tk.x, sb = tk.y, N = pr.nfunc, ta = pr.atom[sa], tb = pr.atom[sb];
  const double wgt = !live ? 0.0 : (sa == sb ? 1.0 : 2.0);
  const double A[3] = {pr.xyz[3 * sa], pr.xyz[3 * sa + 1], pr.xyz[3 * sa + 2]};
  const double AB[3] = {A[0] - pr.xyz[3 * sb], A[1] - pr.xyz[3 * sb + 1], A[2] - pr.xyz[3 * sb + 2]};
  double y[NA * NB], yw[NA * NB], w[NW];
  weight_block<LA, LB>(D, N, pr.ao[sa], pr.ao[sb], y);
  weight_block<LA, LB>(Wm, N, pr.ao[sa], pr.ao[sb], yw);
  lane_weights<LA, LB>(y, AB, w);
  double gA[3] = {0.0, 0.0, 0.0}, gB[3] = {0.0, 0.0, 0.0}, gS[3] = {0.0, 0.0, 0.0};   // gS: overlap on A
  const int np = pr.nprim[sa] * pr.nprim[sb];
  int most = np;   // every lane of the warp makes the same number of passes (shuffles below)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
#pragma unroll 1
  for (int ab = 0; ab < most; ++ab) {
    const double on = ab < np ? 1.0 : 0.0;
    const int pp = min(ab, np - 1), nb = pr.nprim[sb];
    const int ia = pr.pstart[sa] + pp / nb, ib = pr.pstart[sb] + pp % nb;
    const double al = pr.exps[ia], be = pr.exps[ib], cc = on * wgt * pr.coefs[ia] * pr.coefs[ib];
    const Prod d = gauss_prod(al, be, A, AB);
    if (ta != tb) {   // overlap and kinetic energy depend on A - B alone
      double s[3][(LA + 2) * LD];
#pragma unroll
      for (int x = 0; x < 3; ++x)
        overlap_1d<LA + 1, LB + 2, LD>(d.PA[x], d.PA[x] + AB[x], 0.5 * d.ip, x == 0 ? cc * d.K : 1.0, s[x]);
      const double f = 3.14159265358979323846 * d.ip, f3 = f * sqrt(f);
#pragma unroll 1
      for (int at = q; at < NA * NB; at += L) {   // the lanes share out the components
        int c[3], e[3];
        cart_decode(LA, at / NB, c[0], c[1], c[2]);
        cart_decode(LB, at % NB, e[0], e[1], e[2]);
        double s0[3], k0[3], ds[3], dk[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          s0[x] = s[x][c[x] * LD + e[x]];
          k0[x] = second_1d(s[x], LD, c[x], e[x], be);
          ds[x] = 2.0 * al * s[x][(c[x] + 1) * LD + e[x]];
          dk[x] = 2.0 * al * second_1d(s[x], LD, c[x] + 1, e[x], be);
          if (c[x] > 0) {
            ds[x] -= c[x] * s[x][(c[x] - 1) * LD + e[x]];
            dk[x] -= c[x] * second_1d(s[x], LD, c[x] - 1, e[x], be);
          }
        }
        const double wd = -0.5 * f3 * y[at], ws = f3 * yw[at];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const int u = (x + 1) % 3, z = (x + 2) % 3;
          const double uz = s0[u] * s0[z];
          gS[x] = fma(ws, ds[x] * uz, gS[x]);
          const double t = wd * fma(dk[x], uz, ds[x] * fma(k0[u], s0[z], s0[u] * k0[z]));
          gA[x] += t;
          gB[x] -= t;
        }
      }
    }
    // nuclear attraction
    double ks[NK];
#pragma unroll
    for (int i = 0; i < NK; ++i) ks[i] = 0.0;
    const double pref = -6.283185307179586 * d.ip * cc * d.K;
#pragma unroll 1
    for (int c0 = 0; c0 < g.natoms; c0 += L) {
      const int c = min(c0 + q, g.natoms - 1);
      const double z = c0 + q < g.natoms ? (double)g.Z[c] : 0.0;
      const double CP[3] = {g.axyz[3 * c] - d.P[0], g.axyz[3 * c + 1] - d.P[1], g.axyz[3 * c + 2] - d.P[2]};
      double F[E + 1], row[cart_offset(E + 1)];
      lane_boys<E>(0, d.p * fma(CP[0], CP[0], fma(CP[1], CP[1], CP[2] * CP[2])), g.boys, F);
      lane_vrr<E>(F, z * pref, d.PA, CP, 0.5 * d.ip, 1.0, row);
      double U[3] = {0.0, 0.0, 0.0}, V = 0.0;   // U: 2p U_i - D_i
#pragma unroll kUnroll
      for (int l = LA; l <= LA + LB; ++l)
#pragma unroll kUnroll
        for (int a = 0; a <= l; ++a)
#pragma unroll kUnroll
          for (int b = 0; b <= a; ++b) {
            const int e[3] = {l - a, a - b, b};
            const double we = w[ecart(e[0], e[1], e[2]) - OW], wp = 2.0 * d.p * we;
            V = fma(we, row[ecart(e[0], e[1], e[2])], V);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              U[i] = fma(wp, row[ecart(e[0] + (i == 0), e[1] + (i == 1), e[2] + (i == 2))], U[i]);
              if (e[i] > 0)
                U[i] = fma(-e[i] * we, row[ecart(e[0] - (i == 0), e[1] - (i == 1), e[2] - (i == 2))], U[i]);
            }
          }
#pragma unroll
      for (int i = 0; i < NK; ++i) ks[i] += row[O + i];
      // the force on nucleus c over the pairs of the warp, then one atomic each
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        double t = -fma(2.0 * be * AB[i], V, U[i]);
#pragma unroll 1
        for (int o = L; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane < L && c0 + q < g.natoms) atomicAdd(grad_one + 3 * c + i, t);
      }
    }
    double s[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) s[i] = 0.0;
    if constexpr (LA + LB < 5) lane_contract<LA, LB>(ks, y, AB, s);
    else contract_call<LA, LB>(ks, y, AB, s);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      gA[x] += fma(2.0 * al, s[x], s[6 + x] - s[3 + x]);
      gB[x] += fma(2.0 * be, fma(AB[x], s[9], s[x]), -s[6 + x]);
    }
  }
#pragma unroll 1
  for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      gA[x] += __shfl_xor_sync(0xffffffffu, gA[x], o);
      gB[x] += __shfl_xor_sync(0xffffffffu, gB[x], o);
      gS[x] += __shfl_xor_sync(0xffffffffu, gS[x], o);
    }
  if (q != 0 || !live) return;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    atomicAdd(grad_one + 3 * ta + x, gA[x]);
    atomicAdd(grad_one + 3 * tb + x, gB[x]);
    if (ta != tb) {
      atomicAdd(grad_ovl + 3 * ta + x, -gS[x]);
      atomicAdd(grad_ovl + 3 * tb + x, gS[x]);
    }
  }
}

// One warp a block.
__global__ void __launch_bounds__(32, 8) lane_grad_one_kernel(const __grid_constant__ OneArgs g, const double* D,
                                                              const double* W, double* grad_one, double* grad_ovl) {
  LaneChunk ch;
  if (!one_chunk(g, ch)) return;
  RIHF_ONE_CASES(grad_one_tasks, D, W, grad_one, grad_ovl)
}

}  // namespace

void launch_lane_grad_one(const IntegralCtx& ic, const DevShells& prim, const Lane2Tasks& t, int lanes, int natoms,
                          const int* Z, const double* axyz, const double* D, const double* W, double* grad_one, double* grad_ovl) {
  if (t.nchunk <= 0) return;
  lane_grad_one_kernel<<<one_grid(t, lanes), 32, 0, ic.stream>>>(one_args(ic, prim, t, lanes, natoms, Z, axyz), D, W,
                                                                 grad_one, grad_ovl);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

}  // namespace rihf
