// Three-centre integrals (mu nu|P), one lane per shell triple (eri3_lane.cuh).
//
// Bound by the FP64 pipe: about 1.9e8 FP64 instructions a lane set for (H2O)8
// (N = 192, Naux = 848: 0.31 ms at the pipe's rate), 3.8e9 for (H2O)10 in the
// larger basis (N = 580, Naux = 1700: 6.4 ms).  Measured 0.47 and 7.6 ms; the
// warp-cooperative kernel (integrals.cu), with its general electron transfer over
// 8 to 32 lanes a task, takes 5.4 and 119 ms.  Whole triples per lane, and not a
// triple over several lanes, because idle lanes of an FP64 instruction cost as
// much as busy ones and every level of the recursion has another length.
#include "eri3_lane.cuh"

#include <algorithm>

#include "../../include/rihf.h"

namespace rihf {

// The tasks of one chunk, class (LA, LB | lc): lane by lane, 32 consecutive
// tasks at a time, written pair-packed into T.
template <int LA, int LB>
__device__ __noinline__ void lane_eri3_chunk(const LaneGeom* __restrict__ G, long long task0, int n, int lc,
                                             const double* __restrict__ boys) {
  constexpr int E = LA + LB, O = cart_offset(LA), NK = cart_offset(E + 1) - O;
  constexpr int FA = nsph(LA), FB = nsph(LB);
  const int N = G->prim.nfunc;
  const long long npp = (long long)N * (N + 1) / 2;
  const KetTable* tab = G->ket + lc;
  double K[nsph(kMaxLAux) * NK];
#pragma unroll 1
  for (int j = threadIdx.x & 31; j < n; j += 32) {
    const int2 tk = G->tasks[task0 + j];
    const int ip = tk.x, sc = tk.y;
    int sa = G->pairs[ip].a, sb = G->pairs[ip].b;
    if (LA != LB && G->prim.l[sa] != LA) { const int t = sa; sa = sb; sb = t; }
    const double* A = G->prim.xyz + 3 * sa;
    const double* B = G->prim.xyz + 3 * sb;
    const double AB[3] = {A[0] - B[0], A[1] - B[1], A[2] - B[2]};
    const double C[3] = {G->aux.xyz[3 * sc], G->aux.xyz[3 * sc + 1], G->aux.xyz[3 * sc + 2]};
    const int nab = G->prim.nprim[sa] * G->prim.nprim[sb], nc = G->aux.nprim[sc], c0 = G->aux.pstart[sc];
    const PairPrim* pr = G->ptab.pp + G->ptab.off[ip];
#pragma unroll 1
    for (int ab = 0; ab < nab; ++ab) {
      const PairPrim q = pr[ab];
#pragma unroll 1
      for (int pc = 0; pc < nc; ++pc)
        lane_triple<E, LA>(q, G->aux, c0 + pc, C, lc, boys, tab, ab + pc == 0, K);
    }
    const int mu0 = G->prim.ao[sa], nu0 = G->prim.ao[sb];
    const bool diag = LA == LB && sa == sb;
    double* T = G->out + (long long)G->aux.ao[sc] * npp;
#pragma unroll 1
    for (int m = 0; m <= 2 * lc; ++m, T += npp) {
      double k[NK], cart[ncart(LA) * ncart(LB)], half[ncart(LA) * FB], out[FA * FB];
#pragma unroll
      for (int e = 0; e < NK; ++e) k[e] = K[m * NK + e];
      lane_hrr<LA, LB>(k, AB, cart);
#pragma unroll
      for (int ka = 0; ka < ncart(LA); ++ka) lane_sph<LB, true>(cart + ka * ncart(LB), 1, half + ka * FB, 1);
#pragma unroll
      for (int fb = 0; fb < FB; ++fb) lane_sph<LA, true>(half + fb, FB, out + fb, FB);
#pragma unroll
      for (int a = 0; a < FA; ++a)
#pragma unroll
        for (int b = 0; b < FB; ++b)
          if (!diag || b <= a) T[lane_tri(mu0 + a, nu0 + b)] = out[a * FB + b];
    }
  }
}

struct Eri3Chunk {
  const LaneGeom* G;
  LaneChunk ch;
  const double* boys;
  template <int LA, int LB>
  __device__ __forceinline__ void run() const {
    lane_eri3_chunk<LA, LB>(G, ch.task0, ch.n, ch.cls >> 8, boys);
  }
};

template <int GRP>
__global__ void __launch_bounds__(32, kLaneBlocks[GRP])
    lane_eri3_kernel(const __grid_constant__ LaneGeom G0, const LaneGeom* __restrict__ geoms,
                     const long long* __restrict__ off, int ngeom, long long nchunk, int* counter,
                     const double* __restrict__ boys) {
  Eri3Chunk c;
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
  if (g == 0) run(lane_eri3_kernel<0>);
  else if (g == 1) run(lane_eri3_kernel<1>);
  else run(lane_eri3_kernel<2>);
  RIHF_LAUNCH_CHECK();
  if (ic.launches) *ic.launches += 1;
}

void launch_lane_eri3(const IntegralCtx& ic, int sms, const LaneTasks& t) {
  RIHF_CUDA(cudaMemsetAsync(ic.counter, 0, kLaneGroups * sizeof(int), ic.stream));
  for (int g = kLaneGroups - 1; g >= 0; --g) {
    if (t.nchunk[g] == 0) continue;
    LaneGeom G = t.geom;
    G.chunks = t.chunks[g];
    launch_group(ic, sms, g, G, nullptr, nullptr, 0, t.nchunk[g]);
  }
}

long long lane_batch_tables(const IntegralCtx& ic, const std::vector<LaneTasks>& batch, int g, LaneBatchTables& t) {
  const int n = (int)batch.size();
  std::vector<LaneGeom> geoms(n);
  std::vector<long long> off(n + 1, 0);
  for (int i = 0; i < n; ++i) {
    geoms[i] = batch[i].geom;
    geoms[i].chunks = batch[i].chunks[g];
    off[i + 1] = off[i] + batch[i].nchunk[g];
  }
  if (off[n] == 0) return 0;
  RIHF_CUDA(cudaMemcpyAsync(t.geoms + (size_t)g * t.cap, geoms.data(), sizeof(LaneGeom) * n, cudaMemcpyHostToDevice,
                            ic.stream));
  RIHF_CUDA(cudaMemcpyAsync(t.off + (size_t)g * (t.cap + 1), off.data(), sizeof(long long) * (n + 1),
                            cudaMemcpyHostToDevice, ic.stream));
  RIHF_CUDA(cudaStreamSynchronize(ic.stream));   // the host arrays are temporaries
  return off[n];
}

void launch_lane_eri3_batch(const IntegralCtx& ic, int sms, const std::vector<LaneTasks>& batch, LaneBatchTables& t) {
  if (batch.empty()) return;
  if ((int)batch.size() > t.cap) throw RihfError(RIHF_ERR_INVALID_ARG, "launch_lane_eri3_batch: batch tables too small");
  RIHF_CUDA(cudaMemsetAsync(ic.counter, 0, kLaneGroups * sizeof(int), ic.stream));
  for (int g = kLaneGroups - 1; g >= 0; --g) {
    const long long n = lane_batch_tables(ic, batch, g, t);
    if (n == 0) continue;
    launch_group(ic, sms, g, batch[0].geom, t.geoms + (size_t)g * t.cap, t.off + (size_t)g * (t.cap + 1),
                 (int)batch.size(), n);
  }
}

// ------------------------------------------------------------ task lists

// FP64 instructions of a derivative task, roughly: the weight by which chunks
// are sized and ordered.
static double lane_cost(int la, int lb, int lc) {
  const int ne = cart_offset(la + lb + 2);
  double kets = 0.0;
  for (int c = 1; c <= lc; ++c) kets += ncart(c);
  return 80.0 + 3.0 * ne + 2.0 * ne * kets + 6.0 * ne * nsph(lc);
}

void build_lane_tasks(const std::vector<ShellPair>& pairs, const std::vector<int>& lprim, const std::vector<int>& patom,
                      const std::vector<int>& laux, const std::vector<int>& aatom, int sms, std::vector<int2>& tasks,
                      std::vector<LaneChunk> (&chunks)[kLaneGroups]) {
  struct Class {
    int la, lb, lc;
    double cost;
  };
  // pairs by class, in the order of their atom pairs; auxiliary shells by l and atom
  std::vector<int> by_class[kMaxLPrim + 1][kMaxLPrim + 1], by_l[kMaxLAux + 1];
  auto atoms = [&](int p) { return std::make_pair(patom[pairs[p].a], patom[pairs[p].b]); };
  for (int p = 0; p < (int)pairs.size(); ++p) {
    const int x = lprim[pairs[p].a], y = lprim[pairs[p].b];
    by_class[std::max(x, y)][std::min(x, y)].push_back(p);
  }
  for (auto& row : by_class)
    for (auto& v : row) std::stable_sort(v.begin(), v.end(), [&](int p, int q) { return atoms(p) < atoms(q); });
  for (int c = 0; c < (int)laux.size(); ++c) by_l[laux[c]].push_back(c);
  for (auto& v : by_l) std::stable_sort(v.begin(), v.end(), [&](int c, int d) { return aatom[c] < aatom[d]; });
  std::vector<Class> classes;
  double total = 0.0;
  for (int la = 0; la <= kMaxLPrim; ++la)
    for (int lb = 0; lb <= la; ++lb)
      for (int lc = 0; lc <= kMaxLAux; ++lc) {
        if (by_class[la][lb].empty() || by_l[lc].empty()) continue;
        classes.push_back({la, lb, lc, lane_cost(la, lb, lc)});
        total += classes.back().cost * by_class[la][lb].size() * by_l[lc].size();
      }
  std::sort(classes.begin(), classes.end(), [](const Class& x, const Class& y) { return x.cost > y.cost; });
  tasks.clear();
  tasks.reserve(pairs.size() * laux.size());
  for (auto& v : chunks) v.clear();
  // a chunk: up to 8 tasks a lane, about 4000 FP64 instructions of each lane at
  // most, and at least three chunks for every resident warp of the whole list
  const double share = total / (3.0 * sms * kLaneBlocks[1] * 32);
  for (const Class& k : classes) {
    const long long t0 = (long long)tasks.size();
    const std::vector<int>&pv = by_class[k.la][k.lb], &cv = by_l[k.lc];
    for (size_t p0 = 0; p0 < pv.size();) {
      size_t p1 = p0;
      while (p1 < pv.size() && atoms(pv[p1]) == atoms(pv[p0])) ++p1;
      for (size_t c0 = 0; c0 < cv.size();) {
        size_t c1 = c0;
        while (c1 < cv.size() && aatom[cv[c1]] == aatom[cv[c0]]) ++c1;
        for (size_t p = p0; p < p1; ++p)
          for (size_t c = c0; c < c1; ++c) tasks.push_back(make_int2(pv[p], cv[c]));
        c0 = c1;
      }
      p0 = p1;
    }
    const int per = (int)std::max(1.0, std::min(8.0, std::min(share, 4000.0) / k.cost));
    const long long n = (long long)tasks.size() - t0;
    std::vector<LaneChunk>& out = chunks[lane_group(k.la, k.lb)];
    for (long long i = 0; i < n; i += 32 * per)
      out.push_back({t0 + i, (int)std::min<long long>(32 * per, n - i), k.la | k.lb << 4 | k.lc << 8});
  }
  for (auto& v : chunks)
    if ((long long)v.size() > kMaxGroupTasks) throw RihfError(RIHF_ERR_INVALID_ARG, "build_lane_tasks: too many 3-centre tasks");
}

// Nonzero coefficients of the real solid harmonics of degree l.
static double sph_terms(int l) {
  double n = 0.0;
  for (int m = -l; m <= l; ++m)
    for (int x = 0; x <= l; ++x)
      for (int y = 0; y <= l - x; ++y) n += bra_sph(l, m, x, y, l - x - y) != 0.0;
  return n;
}

void lane_flops(const std::vector<ShellPair>& pairs, const std::vector<int>& lprim, const std::vector<int>& nprim,
                const std::vector<int>& patom, const std::vector<int>& laux, const std::vector<int>& naux_prim,
                const std::vector<int>& aatom, const std::vector<KetTable>& ket, double* eri3, double* grad3) {
  // one primitive triple: setup, Boys step, bra recursion, ket steps and their sums into the harmonics
  auto triple = [&](int E, int emin, int lc) {
    double f = 60.0 + 12.0 * (E + 1) + (E + 1);
    for (int l = 1; l <= E; ++l)
      for (int a = 0; a <= l; ++a)
        for (int b = 0; b <= a; ++b) {
          const int x = l - a, y = a - b, z = b, n = (x > 0 ? x : y > 0 ? y : z) - 1;
          f += (E - l + 1) * (n > 0 ? 7.0 : 3.0);
        }
    for (int s = 1; s <= lc; ++s)
      for (int l = std::max(0, emin - (lc - s)); l <= E; ++l)   // components x: ncart(s); e_i > 0: two of three on average
        f += ncart(s) * (ncart(l) + 2.0 * (l > 0 ? ncart(l - 1) : 0));
    const double ne = cart_offset(E + 1) - cart_offset(emin);
    return f + (lc > 1 ? 2.0 * ne * ket[lc].start[ncart(lc)] : 0.0);
  };
  auto hrr = [](int la, int lb) {
    double f = 0.0;
    for (int b = 1; b <= lb; ++b) f += 2.0 * (cart_offset(la + lb - b + 1) - cart_offset(la)) * ncart(b);
    return f;
  };
  auto bra = [&](int la, int lb) {   // one spherical transform of a Cartesian (la, lb) block
    return 2.0 * ((lb > 1 ? ncart(la) * sph_terms(lb) : 0.0) + (la > 1 ? nsph(lb) * sph_terms(la) : 0.0));
  };
  double e3[kMaxLPrim + 1][kMaxLPrim + 1][kMaxLAux + 1], e1[kMaxLPrim + 1][kMaxLPrim + 1][kMaxLAux + 1];
  double g3[kMaxLPrim + 1][kMaxLPrim + 1][kMaxLAux + 1], g1[kMaxLPrim + 1][kMaxLPrim + 1][kMaxLAux + 1];
  for (int la = 0; la <= kMaxLPrim; ++la)
    for (int lb = 0; lb <= la; ++lb)
      for (int lc = 0; lc <= kMaxLAux; ++lc) {
        e3[la][lb][lc] = triple(la + lb, la, lc);
        e1[la][lb][lc] = nsph(lc) * (hrr(la, lb) + bra(la, lb));
        g3[la][lb][lc] = triple(la + lb + 1, la > 0 ? la - 1 : 0, lc);
        const double nw = cart_offset(la + lb + 1) - cart_offset(la);
        double f = bra(la, lb) + hrr(la, lb) + 8.0 * nw;
        for (int l = std::max(la, 1); l <= la + lb; ++l) f += 6.0 * ncart(l - 1);
        if (lb > 0) f += hrr(la, lb - 1) + 6.0 * ncart(la) * ncart(lb - 1);
        g1[la][lb][lc] = nsph(lc) * f + 30.0;
      }
  double fe = 0.0, fg = 0.0;
  for (const ShellPair& sp : pairs) {
    int a = sp.a, b = sp.b;
    if (lprim[a] < lprim[b]) std::swap(a, b);
    const double nab = (double)nprim[a] * nprim[b];
    for (int c = 0; c < (int)laux.size(); ++c) {
      const int la = lprim[a], lb = lprim[b], lc = laux[c];
      fe += nab * naux_prim[c] * e3[la][lb][lc] + e1[la][lb][lc];
      if (patom[a] != patom[b] || patom[b] != aatom[c]) fg += nab * (naux_prim[c] * g3[la][lb][lc] + g1[la][lb][lc]);
    }
  }
  *eri3 = fe;
  *grad3 = fg;
}

std::vector<KetTable> build_ket_tables(const std::vector<double>& tr, const std::vector<int>& nf) {
  std::vector<KetTable> out(kMaxLAux + 1);
  for (int l = 0; l <= kMaxLAux; ++l) {
    KetTable& t = out[l];
    int n = 0, v = 0;
    std::vector<char> seen(nf[l], 0);
    for (int cx = 0; cx <= l; ++cx)
      for (int cy = 0; cy <= l - cx; ++cy) {
        t.start[v++] = n;
        for (int m = 0; m < nf[l]; ++m) {
          const double c = tr[(size_t)l * kTrStride * kTrStride + m * kTrStride + kcart(cx, cy, l - cx - cy)];
          if (c == 0.0) continue;
          t.term[n++] = {c, m, seen[m] ? 0 : 1};
          seen[m] = 1;
        }
      }
    for (; v <= ncart(kMaxLAux); ++v) t.start[v] = n;
  }
  return out;
}

}  // namespace rihf
