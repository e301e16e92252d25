// One-electron integrals for spherical bases: 4 to 32 lanes per shell pair, which
// share out the nuclei (the recursion of eri3_lane.cuh with a point-charge ket, i.e.
// no ket steps; how many lanes: one_lanes).  Measured 0.077 ms at (H2O)8 (4656
// pairs, 24 nuclei), 0.38 ms at (H2O)10 in the larger basis; the warp-cooperative
// kernel takes 0.39 and 3.1 ms.
#include <algorithm>

#include "../../include/rihf.h"
#include "one_lane.cuh"

namespace rihf {

namespace {

template <int LA, int LB>
__device__ __noinline__ void one_tasks(const OneArgs& g, const LaneChunk& ch, double* __restrict__ S, double* __restrict__ H) {
  constexpr int E = LA + LB, O = cart_offset(LA), NK = cart_offset(E + 1) - O;
  constexpr int NA = ncart(LA), NB = ncart(LB), FA = nsph(LA), FB = nsph(LB), LD = LB + 3;
  const int L = g.lanes, q = threadIdx.x & (L - 1), slot = threadIdx.x >> (31 - __clz(L));
  const int j = min(slot, ch.n - 1);   // idle lanes repeat the last
  const DevShells& pr = g.prim;
  const int2 tk = g.tasks[ch.task0 + j];
  const int sa = tk.x, sb = tk.y, N = pr.nfunc;
  const double A[3] = {pr.xyz[3 * sa], pr.xyz[3 * sa + 1], pr.xyz[3 * sa + 2]};
  const double AB[3] = {A[0] - pr.xyz[3 * sb], A[1] - pr.xyz[3 * sb + 1], A[2] - pr.xyz[3 * sb + 2]};
  double k[NK], sc[NA * NB], tc[NA * NB];
#pragma unroll
  for (int e = 0; e < NK; ++e) k[e] = 0.0;
#pragma unroll
  for (int e = 0; e < NA * NB; ++e) sc[e] = tc[e] = 0.0;
#pragma unroll 1
  for (int pa = 0; pa < pr.nprim[sa]; ++pa)
#pragma unroll 1
    for (int pb = 0; pb < pr.nprim[sb]; ++pb) {
      const int ia = pr.pstart[sa] + pa, ib = pr.pstart[sb] + pb;
      const double be = pr.exps[ib], w = pr.coefs[ia] * pr.coefs[ib];
      const Prod d = gauss_prod(pr.exps[ia], be, A, AB);
      double s[3][(LA + 1) * LD], kd[3][(LA + 1) * (LB + 1)];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        overlap_1d<LA, LB + 2, LD>(d.PA[x], d.PA[x] + AB[x], 0.5 * d.ip, x == 0 ? w * d.K : 1.0, s[x]);
#pragma unroll
        for (int i = 0; i <= LA; ++i)
#pragma unroll
          for (int l = 0; l <= LB; ++l) kd[x][i * (LB + 1) + l] = -0.5 * second_1d(s[x], LD, i, l, be);
      }
      const double f = 3.14159265358979323846 * d.ip, f3 = f * sqrt(f);   // the three sqrt(pi / p)
#pragma unroll
      for (int a = 0; a <= LA; ++a)
#pragma unroll
        for (int c = 0; c <= a; ++c)
#pragma unroll
          for (int b = 0; b <= LB; ++b)
#pragma unroll
            for (int e = 0; e <= b; ++e) {
              const int ca[3] = {LA - a, a - c, c}, cb[3] = {LB - b, b - e, e};
              const int at = kcart(ca[0], ca[1], ca[2]) * NB + kcart(cb[0], cb[1], cb[2]);
              double sx[3], kx[3];
#pragma unroll
              for (int x = 0; x < 3; ++x) {
                sx[x] = s[x][ca[x] * LD + cb[x]];
                kx[x] = kd[x][ca[x] * (LB + 1) + cb[x]];
              }
              const double yz = sx[1] * sx[2];
              sc[at] = fma(f3, sx[0] * yz, sc[at]);
              tc[at] = fma(f3, fma(kx[0], yz, sx[0] * fma(kx[1], sx[2], sx[1] * kx[2])), tc[at]);
            }
      const double pref = 6.283185307179586 * d.ip * w * d.K;
#pragma unroll 1
      for (int c = q; c < g.natoms; c += L) {
        const double CP[3] = {g.axyz[3 * c] - d.P[0], g.axyz[3 * c + 1] - d.P[1], g.axyz[3 * c + 2] - d.P[2]};
        double F[E + 1], row[cart_offset(E + 1)];
        lane_boys<E>(0, d.p * fma(CP[0], CP[0], fma(CP[1], CP[1], CP[2] * CP[2])), g.boys, F);
        lane_vrr<E>(F, -(double)g.Z[c] * pref, d.PA, CP, 0.5 * d.ip, 1.0, row);
#pragma unroll
        for (int e = 0; e < NK; ++e) k[e] += row[O + e];
      }
    }
#pragma unroll 1
  for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
    for (int e = 0; e < NK; ++e) k[e] += __shfl_xor_sync(0xffffffffu, k[e], o);
  if (q != 0 || slot >= ch.n) return;
  double v[NA * NB], out[FA * FB];
  lane_hrr<LA, LB>(k, AB, v);
#pragma unroll
  for (int e = 0; e < NA * NB; ++e) v[e] += tc[e];
  const int mu0 = pr.ao[sa], nu0 = pr.ao[sb];
  auto store = [&](double* M) {
#pragma unroll
    for (int a = 0; a < FA; ++a)
#pragma unroll
      for (int b = 0; b < FB; ++b) {
        M[(size_t)(mu0 + a) * N + nu0 + b] = out[a * FB + b];
        M[(size_t)(nu0 + b) * N + mu0 + a] = out[a * FB + b];
      }
  };
  bra_block<LA, LB>(v, out);
  store(H);
  bra_block<LA, LB>(sc, out);
  store(S);
}

// One warp a block.
__global__ void __launch_bounds__(32, 8) lane_one_kernel(const __grid_constant__ OneArgs g, double* S, double* H) {
  LaneChunk ch;
  if (!one_chunk(g, ch)) return;
  RIHF_ONE_CASES(one_tasks, S, H)
}
}  // namespace

// The lanes of a pair: the most that leave at most 32 warps an SM.  Below that the
// latency of one pair's chain over the nuclei is the time, and more lanes shorten it;
// above, FP64 instructions count and the part of a pair that every lane repeats makes
// more lanes dearer (contexts of a batch launch beside each other, and each gets
// its share: 16 of 3 to 6 waters take 0.7 ms longer in 102 when each fills the SMs by
// itself).  No more than about two a nucleus (the components that the
// derivative also shares out use the second): with three nuclei in the larger basis 32
// lanes make the integrals 0.125 ms, 8 lanes 0.119.  Derivatives with 4 / 8 / 16 / 32 lanes: (H2O)3, 666 pairs, 0.176 /
// 0.135 / 0.100 / 0.084 ms; (H2O)8, 4656 pairs, 0.268 / 0.176 / 0.143 / 0.139; (H2O)12,
// 10440 pairs, 0.397 / 0.276 / 0.272 / 0.387.
int one_lanes(int nshell, int natoms, int sms, int share) {
  const long long pairs = (long long)nshell * (nshell + 1) / 2 * share;
  int lanes = 4;
  while (lanes < 32 && lanes < 2 * natoms) lanes *= 2;
  while (lanes > 4 && pairs * lanes > 32LL * 32 * sms) lanes /= 2;
  return lanes;
}

void build_one_tasks(const std::vector<int>& l, std::vector<int2>& tasks, std::vector<LaneChunk>& chunks) {
  std::vector<int> by_l[kMaxLPrim + 1];
  for (int i = 0; i < (int)l.size(); ++i) by_l[l[i]].push_back(i);
  tasks.clear();
  chunks.clear();
  for (int la = kMaxLPrim; la >= 0; --la)   // heavy classes first
    for (int lb = la; lb >= 0; --lb) {
      const long long t0 = (long long)tasks.size();
      for (int a : by_l[la])
        for (int b : by_l[lb])
          if (la != lb || a >= b) tasks.push_back(make_int2(a, b));
      const long long n = (long long)tasks.size() - t0;
      for (long long i = 0; i < n; i += kOneChunk)
        chunks.push_back({t0 + i, (int)std::min<long long>(kOneChunk, n - i), la | lb << 4});
    }
}

void launch_lane_one(const IntegralCtx& ic, const DevShells& prim, const Lane2Tasks& t, int lanes, int natoms, const int* Z,
                     const double* axyz, double* S, double* H) {
  if (t.nchunk <= 0) return;
  lane_one_kernel<<<one_grid(t, lanes), 32, 0, ic.stream>>>(one_args(ic, prim, t, lanes, natoms, Z, axyz), S, H);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

}  // namespace rihf
