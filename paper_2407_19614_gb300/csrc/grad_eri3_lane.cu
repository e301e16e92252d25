// Fused three-centre derivative contraction sum Y d(mu nu|P), one lane per shell
// triple (eri3_lane.cuh).
//
// With w[e] = sum_ab Y_ab binom(b, e - a) AB^(b - e + a), the horizontal
// recurrence applied to Y instead of the integrals, every derivative term of a
// triple is a short sum over [e|l m], e in [la - 1, la + lb + 1]:
//   U_i = sum_ab Y (a+1_i b| = sum_e w[e] [e+1_i|,   V = sum_e w[e] [e|,
//   D_i = sum_e e_i w[e] [e-1_i|,   B_i = sum_ab b_i Y (a b-1_i|,
//   dE/dA_i = 2 alpha U_i - D_i + B_i  (sum_ab a_i Y (a-1_i b| = D_i - B_i),
//   dE/dB_i = 2 beta (U_i + AB_i V) - B_i,   dE/dC = -(dE/dA + dE/dB),
// so only (a b-1| runs a recurrence on the integrals.
//
// Bound by the FP64 pipe: 4.7e8 FP64 instructions a lane set for (H2O)8 (0.78 ms
// at its rate), 9.5e9 for (H2O)10 in the larger basis (15.9 ms).  Measured 1.30
// and 19.5 ms; the warp-cooperative kernel with its four recurrences
// (grad_integrals.cu) takes 11.2 and 251 ms.
#include <algorithm>

#include "../../include/rihf.h"
#include "grad_lane.cuh"

namespace rihf {

// The tasks of one chunk, class (LA, LB | lc): every lane takes a run of
// consecutive tasks and keeps its sums while the three atoms stay the same.
template <int LA, int LB>
__device__ __noinline__ void lane_grad_chunk(const LaneGeom* __restrict__ G, long long task0, int n, int lc,
                                             const double* __restrict__ boys) {
  constexpr int E = LA + LB + 1, EMIN = LA > 0 ? LA - 1 : 0, NK = cart_offset(E + 1) - cart_offset(EMIN);
  constexpr int FA = nsph(LA), FB = nsph(LB);
  const int N = G->prim.nfunc;
  const long long npp = (long long)N * (N + 1) / 2;
  const KetTable* tab = G->ket + lc;
  double K[nsph(kMaxLAux) * NK];
  const int run = (n + 31) / 32, j0 = (threadIdx.x & 31) * run, j1 = min(n, j0 + run);
  int at[3] = {-1, -1, -1};
  double g[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  auto flush = [&]() {
    if (at[0] < 0) return;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      atomicAdd(G->out + 3 * at[0] + x, g[x]);
      atomicAdd(G->out + 3 * at[1] + x, g[3 + x]);
      atomicAdd(G->out + 3 * at[2] + x, -(g[x] + g[3 + x]));
      g[x] = g[3 + x] = 0.0;
    }
  };
#pragma unroll 1
  for (int j = j0; j < j1; ++j) {
    const int2 tk = G->tasks[task0 + j];
    const int ip = tk.x, sc = tk.y;
    int sa = G->pairs[ip].a, sb = G->pairs[ip].b;
    if (LA != LB && G->prim.l[sa] != LA) { const int t = sa; sa = sb; sb = t; }   // Y is symmetric
    const int ta = G->prim.atom[sa], tb = G->prim.atom[sb], tc = G->aux.atom[sc];
    if (ta == tb && tb == tc) continue;   // one centre: the derivatives sum to zero
    if (ta != at[0] || tb != at[1] || tc != at[2]) {
      flush();
      at[0] = ta;
      at[1] = tb;
      at[2] = tc;
    }
    const double* A = G->prim.xyz + 3 * sa;
    const double* B = G->prim.xyz + 3 * sb;
    const double AB[3] = {A[0] - B[0], A[1] - B[1], A[2] - B[2]};
    const double C[3] = {G->aux.xyz[3 * sc], G->aux.xyz[3 * sc + 1], G->aux.xyz[3 * sc + 2]};
    const int nab = G->prim.nprim[sa] * G->prim.nprim[sb], nc = G->aux.nprim[sc], c0 = G->aux.pstart[sc];
    const PairPrim* pr = G->ptab.pp + G->ptab.off[ip];
    const int mu0 = G->prim.ao[sa], nu0 = G->prim.ao[sb];
    const double wgt = sa == sb ? 1.0 : 2.0;
    const double* Yc = G->Y + (long long)G->aux.ao[sc] * npp;
#pragma unroll 1
    for (int ab = 0; ab < nab; ++ab) {
      double al, be;
      {
        const PairPrim q = pr[ab];
        al = q.alpha;
        be = q.beta;
#pragma unroll 1
        for (int pc = 0; pc < nc; ++pc) lane_triple<E, EMIN>(q, G->aux, c0 + pc, C, lc, boys, tab, pc == 0, K);
      }
      double s[10];
#pragma unroll
      for (int i = 0; i < 10; ++i) s[i] = 0.0;
#pragma unroll 1
      for (int m = 0; m <= 2 * lc; ++m) {
        double y[FA * FB], half[ncart(LA) * FB], yc[ncart(LA) * ncart(LB)], k[NK];
#pragma unroll
        for (int a = 0; a < FA; ++a)
#pragma unroll
          for (int b = 0; b < FB; ++b) y[a * FB + b] = __ldg(Yc + m * npp + lane_tri(mu0 + a, nu0 + b));
#pragma unroll
        for (int e = 0; e < NK; ++e) k[e] = K[m * NK + e];
#pragma unroll
        for (int b = 0; b < FB; ++b) lane_sph<LA, false>(y + b, FB, half + b, FB);
#pragma unroll
        for (int ka = 0; ka < ncart(LA); ++ka) lane_sph<LB, false>(half + ka * FB, 1, yc + ka * ncart(LB), 1);
        lane_contract<LA, LB>(k, yc, AB, s);
      }
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        g[x] = fma(wgt, fma(2.0 * al, s[x], s[6 + x] - s[3 + x]), g[x]);
        g[3 + x] = fma(wgt, fma(2.0 * be, fma(AB[x], s[9], s[x]), -s[6 + x]), g[3 + x]);
      }
    }
  }
  flush();
}

struct GradChunk {
  const LaneGeom* G;
  LaneChunk ch;
  const double* boys;
  template <int LA, int LB>
  __device__ __forceinline__ void run() const {
    lane_grad_chunk<LA, LB>(G, ch.task0, ch.n, ch.cls >> 8, boys);
  }
};

template <int GRP>
__global__ void __launch_bounds__(32, kLaneBlocks[GRP])
    lane_grad_kernel(const __grid_constant__ LaneGeom G0, const LaneGeom* __restrict__ geoms,
                     const long long* __restrict__ off, int ngeom, long long nchunk, int* counter,
                     const double* __restrict__ boys) {
  GradChunk c;
  c.boys = boys;
  while (lane_claim(G0, geoms, off, ngeom, nchunk, counter, c.G, c.ch)) {
    lane_dispatch<GRP>(c.ch.cls, c);
    __syncwarp();
  }
}

// ------------------------------------------------------------ launchers

static void launch_group(const IntegralCtx& ic, int sms, int g, const LaneGeom& G0, const LaneGeom* geoms,
                         const long long* off, int ngeom, long long nchunk) {
  const int grid = (int)std::min<long long>(nchunk, (long long)sms * kLaneBlocks[g]);
  auto run = [&](auto kernel) {
    kernel<<<grid, 32, 0, ic.stream>>>(G0, geoms, off, ngeom, nchunk, ic.counter + g, ic.boys);
  };
  if (g == 0) run(lane_grad_kernel<0>);
  else if (g == 1) run(lane_grad_kernel<1>);
  else run(lane_grad_kernel<2>);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

void launch_lane_grad(const IntegralCtx& ic, int sms, const LaneTasks& t) {
  RIHF_CUDA(cudaMemsetAsync(ic.counter, 0, kLaneGroups * sizeof(int), ic.stream));
  for (int g = kLaneGroups - 1; g >= 0; --g) {
    if (t.nchunk[g] == 0) continue;
    LaneGeom G = t.geom;
    G.chunks = t.chunks[g];
    launch_group(ic, sms, g, G, nullptr, nullptr, 0, t.nchunk[g]);
  }
}

void launch_lane_grad_batch(const IntegralCtx& ic, int sms, const std::vector<LaneTasks>& batch, LaneBatchTables& t) {
  if (batch.empty()) return;
  if ((int)batch.size() > t.cap) throw RihfError(RIHF_ERR_INVALID_ARG, "launch_lane_grad_batch: batch tables too small");
  RIHF_CUDA(cudaMemsetAsync(ic.counter, 0, kLaneGroups * sizeof(int), ic.stream));
  for (int g = kLaneGroups - 1; g >= 0; --g) {
    const long long n = lane_batch_tables(ic, batch, g, t);
    if (n == 0) continue;
    launch_group(ic, sms, g, batch[0].geom, t.geoms + (size_t)g * t.cap, t.off + (size_t)g * (t.cap + 1),
                 (int)batch.size(), n);
  }
}

}  // namespace rihf
