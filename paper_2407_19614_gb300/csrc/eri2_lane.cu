// (P|Q) and its derivative contraction, one lane per shell pair (eri3_lane.cuh):
// the shell of lower l is the bra, a single function in place of a pair (zero
// exponent on b), so the bra recursion stays short and the two-term ket steps do
// most of the work.
//
// Bound by FP64 instructions and, below a few thousand tasks, by the latency of one
// task.  (H2O)8 (304 auxiliary shells, 46360 tasks): 0.05 and 0.13 ms, against 0.52
// and 0.76 ms of the warp-cooperative kernels; (H2O)10 in the larger basis 0.12 and
// 0.33 ms against 2.6 and 3.9.
#include <algorithm>

#include "../../include/rihf.h"
#include "grad_lane.cuh"
#include "lane2.cuh"

namespace rihf {

namespace {

// One auxiliary primitive as a bra pair with a unit function of zero exponent.
__device__ __forceinline__ PairPrim single_bra(const DevShells& aux, int ia, const double (&A)[3]) {
  PairPrim q;
  const double ip = aux.iexps[ia];
  q.p = q.alpha = aux.exps[ia];
  q.inv_p = ip;
  q.beta = 0.0;
  q.K = 34.98683665524972 * aux.coefs[ia] * ip;   // 2 pi^{5/2} c / p
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q.P[i] = A[i];
    q.PA[i] = 0.0;
  }
  return q;
}

template <int LA>
__device__ __noinline__ void eri2_tasks(const DevShells& aux, const int2* __restrict__ tasks, const LaneChunk& ch,
                                        const KetTable* __restrict__ ket, const double* __restrict__ boys,
                                        double* __restrict__ Am) {
  constexpr int FA = nsph(LA), NK = ncart(LA);
  const int lc = ch.cls >> 8, j = threadIdx.x;
  if (j >= ch.n) return;
  const int2 tk = tasks[ch.task0 + j];
  const int sa = tk.x, sc = tk.y, NA = aux.nfunc;
  const double A[3] = {aux.xyz[3 * sa], aux.xyz[3 * sa + 1], aux.xyz[3 * sa + 2]};
  const double C[3] = {aux.xyz[3 * sc], aux.xyz[3 * sc + 1], aux.xyz[3 * sc + 2]};
  double K[nsph(kMaxLAux) * NK];
  for (int pa = 0; pa < aux.nprim[sa]; ++pa) {
    const PairPrim q = single_bra(aux, aux.pstart[sa] + pa, A);
    for (int pc = 0; pc < aux.nprim[sc]; ++pc)
      lane_triple<LA, LA>(q, aux, aux.pstart[sc] + pc, C, lc, boys, ket + lc, pa + pc == 0, K);
  }
  const int P0 = aux.ao[sa], Q0 = aux.ao[sc];
#pragma unroll 1
  for (int m = 0; m <= 2 * lc; ++m) {
    double k[NK], out[FA];
#pragma unroll
    for (int e = 0; e < NK; ++e) k[e] = K[m * NK + e];
    lane_sph<LA, true>(k, 1, out, 1);
#pragma unroll
    for (int a = 0; a < FA; ++a) {
      Am[(size_t)(P0 + a) * NA + Q0 + m] = out[a];
      Am[(size_t)(Q0 + m) * NA + P0 + a] = out[a];
    }
  }
}

template <int LA>
__device__ __noinline__ void grad_eri2_tasks(const DevShells& aux, const int2* __restrict__ tasks, const LaneChunk& ch,
                                             const KetTable* __restrict__ ket, const double* __restrict__ boys,
                                             const double* __restrict__ Z, double* grad) {
  constexpr int E = LA + 1, EMIN = LA > 0 ? LA - 1 : 0, NK = cart_offset(E + 1) - cart_offset(EMIN), FA = nsph(LA);
  const int lc = ch.cls >> 8, j = threadIdx.x;
  int ta = -1, tc = -1;
  double g[3] = {0.0, 0.0, 0.0};
  if (j < ch.n) {
    const int2 tk = tasks[ch.task0 + j];
    const int sa = tk.x, sc = tk.y, NA = aux.nfunc;
    ta = aux.atom[sa];
    tc = aux.atom[sc];
    if (ta != tc) {   // (P|Q) of one atom does not move
      const double A[3] = {aux.xyz[3 * sa], aux.xyz[3 * sa + 1], aux.xyz[3 * sa + 2]};
      const double C[3] = {aux.xyz[3 * sc], aux.xyz[3 * sc + 1], aux.xyz[3 * sc + 2]};
      const double AB[3] = {0.0, 0.0, 0.0};
      double K[nsph(kMaxLAux) * NK];
      for (int pa = 0; pa < aux.nprim[sa]; ++pa) {
        const PairPrim q = single_bra(aux, aux.pstart[sa] + pa, A);
        for (int pc = 0; pc < aux.nprim[sc]; ++pc)
          lane_triple<E, EMIN>(q, aux, aux.pstart[sc] + pc, C, lc, boys, ket + lc, pc == 0, K);
        double s[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) s[i] = 0.0;
#pragma unroll 1
        for (int m = 0; m <= 2 * lc; ++m) {
          double z[FA], zc[ncart(LA)], k[NK];
#pragma unroll
          for (int a = 0; a < FA; ++a) z[a] = __ldg(Z + (size_t)(aux.ao[sa] + a) * NA + aux.ao[sc] + m);
#pragma unroll
          for (int e = 0; e < NK; ++e) k[e] = K[m * NK + e];
          lane_sph<LA, false>(z, 1, zc, 1);
          lane_contract<LA, 0>(k, zc, AB, s);
        }
        // -1/2 over ordered pairs: every unordered one counts twice
#pragma unroll
        for (int x = 0; x < 3; ++x) g[x] -= fma(2.0 * q.alpha, s[x], -s[3 + x]);
      }
    }
  }
  // tasks come by atom pair: a warp of one pair adds up before its atomics
  const int ta0 = __shfl_sync(0xffffffffu, ta, 0), tc0 = __shfl_sync(0xffffffffu, tc, 0);
  const bool one = __all_sync(0xffffffffu, j >= ch.n || (ta == ta0 && tc == tc0));
  if (one) {
#pragma unroll
    for (int x = 0; x < 3; ++x)
      for (int o = 16; o > 0; o >>= 1) g[x] += __shfl_xor_sync(0xffffffffu, g[x], o);
    if (j > 0) return;
  }
  if (j >= ch.n || ta == tc) return;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    atomicAdd(grad + 3 * ta + x, g[x]);
    atomicAdd(grad + 3 * tc + x, -g[x]);
  }
}

// One block (warp) per chunk.
__global__ void __launch_bounds__(32, 8) lane_eri2_kernel(const __grid_constant__ DevShells aux, const int2* tasks,
                                                          const LaneChunk* chunks, const KetTable* ket,
                                                          const double* boys, double* Am) {
  const LaneChunk ch = chunks[blockIdx.x];
  switch (ch.cls & 0xf) {
    case 0: eri2_tasks<0>(aux, tasks, ch, ket, boys, Am); break;
    case 1: eri2_tasks<1>(aux, tasks, ch, ket, boys, Am); break;
    case 2: eri2_tasks<2>(aux, tasks, ch, ket, boys, Am); break;
    case 3: eri2_tasks<3>(aux, tasks, ch, ket, boys, Am); break;
    default: eri2_tasks<4>(aux, tasks, ch, ket, boys, Am); break;
  }
}

__global__ void __launch_bounds__(32, 8) lane_grad_eri2_kernel(const __grid_constant__ DevShells aux, const int2* tasks,
                                                               const LaneChunk* chunks, const KetTable* ket,
                                                               const double* boys, const double* Z, double* grad) {
  const LaneChunk ch = chunks[blockIdx.x];
  switch (ch.cls & 0xf) {
    case 0: grad_eri2_tasks<0>(aux, tasks, ch, ket, boys, Z, grad); break;
    case 1: grad_eri2_tasks<1>(aux, tasks, ch, ket, boys, Z, grad); break;
    case 2: grad_eri2_tasks<2>(aux, tasks, ch, ket, boys, Z, grad); break;
    case 3: grad_eri2_tasks<3>(aux, tasks, ch, ket, boys, Z, grad); break;
    default: grad_eri2_tasks<4>(aux, tasks, ch, ket, boys, Z, grad); break;
  }
}

}  // namespace

void build_lane2_tasks(const std::vector<int>& l, const std::vector<int>& atom, std::vector<int2>& tasks,
                       std::vector<LaneChunk>& chunks) {
  std::vector<int> by_l[kMaxLAux + 1];
  for (int i = 0; i < (int)l.size(); ++i) by_l[l[i]].push_back(i);
  for (auto& v : by_l) std::stable_sort(v.begin(), v.end(), [&](int a, int b) { return atom[a] < atom[b]; });
  tasks.clear();
  chunks.clear();
  for (int la = kMaxLAux; la >= 0; --la)   // heavy classes first
    for (int lc = kMaxLAux; lc >= la; --lc) {
      const long long t0 = (long long)tasks.size();
      const std::vector<int>&va = by_l[la], &vc = by_l[lc];
      for (size_t a0 = 0; a0 < va.size();) {   // atom pair by atom pair
        size_t a1 = a0;
        while (a1 < va.size() && atom[va[a1]] == atom[va[a0]]) ++a1;
        for (size_t c0 = 0; c0 < vc.size();) {
          size_t c1 = c0;
          while (c1 < vc.size() && atom[vc[c1]] == atom[vc[c0]]) ++c1;
          for (size_t a = a0; a < a1; ++a)
            for (size_t c = c0; c < c1; ++c)
              if (la != lc || va[a] >= vc[c]) tasks.push_back(make_int2(va[a], vc[c]));
          c0 = c1;
        }
        a0 = a1;
      }
      const long long n = (long long)tasks.size() - t0;
      for (long long i = 0; i < n; i += 32) chunks.push_back({t0 + i, (int)std::min<long long>(32, n - i), la | lc << 8});
    }
}

void launch_lane_eri2(const IntegralCtx& ic, const DevShells& aux, const Lane2Tasks& t, const KetTable* ket, double* A) {
  if (t.nchunk <= 0) return;
  lane_eri2_kernel<<<(unsigned)t.nchunk, 32, 0, ic.stream>>>(aux, t.tasks, t.chunks, ket, ic.boys, A);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

void launch_lane_grad_eri2(const IntegralCtx& ic, const DevShells& aux, const Lane2Tasks& t, const KetTable* ket,
                           const double* Z, double* grad) {
  if (t.nchunk <= 0) return;
  lane_grad_eri2_kernel<<<(unsigned)t.nchunk, 32, 0, ic.stream>>>(aux, t.tasks, t.chunks, ket, ic.boys, Z, grad);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

}  // namespace rihf
