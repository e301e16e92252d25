// Walks every address that the FP64 GEMM forms (gemm_index.cuh, the kernel's own
// functions), block by block and thread by thread, over shapes on both sides of its
// tiles, chunks and slices:
//  * each copy reads inside its operand and writes inside its stage of the ring, and
//    the copies of a chunk cover exactly the elements that the chunk's products read;
//  * over all slices, each (m, n, batch, k) product is formed once;
//  * the results of a tile, stored directly, through the cluster's parts or through
//    the workspace, lie inside C and the workspace, and each element of C has one
//    writer (with `mirror`, of both triangles);
//  * the launch is legal: a cluster of 2 to 8 blocks that divides the grid.
// Prints "OK" and exits 0, or names the first violations and exits 1.
#include "gemm_index.cuh"

#include <cstdio>
#include <map>
#include <vector>

using namespace rihf;

namespace {

int g_fail = 0;
const GemmArgs* g_now = nullptr;

void expect(bool ok, const char* what) {
  if (ok || g_fail++ >= 20) return;
  printf("M %d N %d K %d batch %d reduce %d lower %d mirror %d tA %d tB %d: %s\n", g_now->M, g_now->N, g_now->K,
         g_now->batch, g_now->reduce_batch, g_now->lower_only, g_now->mirror, g_now->transA, g_now->transB, what);
}

template <bool TA, bool TB>
void walk(const GemmArgs& g, const GemmPlan& p, size_t work_elems) {
  const int nb = g.reduce_batch ? 1 : g.batch;
  // extents of the operands, the last row without its padding
  const long long extA = (long long)(g.batch - 1) * g.sA + (TA ? (long long)(g.K - 1) * g.lda + g.M : (long long)(g.M - 1) * g.lda + g.K);
  const long long extB = (long long)(g.batch - 1) * g.sB + (TB ? (long long)(g.N - 1) * g.ldb + g.K : (long long)(g.K - 1) * g.ldb + g.N);
  const long long extC = (long long)(nb - 1) * g.sC + (long long)(g.M - 1) * g.ldc + g.N;
  std::vector<int> writers(extC, 0);
  std::vector<long long> ks((size_t)p.ctas, 0);   // products' k summed over the slices, by tile and batch
  for (long long bx = 0; bx < p.ctas; ++bx)
    for (int by = 0; by < p.nslice; ++by) {
      const GemmBlock q = gemm_block(g, (int)bx, by, p.tiles, p.tn, p.kper, p.bper, p.chunk);
      expect(q.batch < nb && q.m0 < g.M && q.n0 < g.N && q.m0 >= 0 && q.n0 >= 0, "tile outside the result");
      expect(g.K == 0 || q.total > 0, "slice without work");
      for (int c = 0; c < q.total; ++c) {
        const int b = q.b0 + c / q.per, kc = q.k0 + (c % q.per) * p.chunk, kv = std::min(p.chunk, q.k1 - kc);
        expect(b < g.batch && kv > 0 && kv <= GK, "chunk outside its slice");
        bool a_in[GK][GT] = {}, b_in[GK][GT] = {};
        for (int tid = 0; tid < GThreads; ++tid)
          for (int idx = tid; idx < GT * p.chunk; idx += GThreads) {
            const GemmElem a = gemm_elem<!TA>(idx, p.chunk, q.m0, g.M, kc, q.k1, g.lda);
            const GemmElem e = gemm_elem<TB>(idx, p.chunk, q.n0, g.N, kc, q.k1, g.ldb);
            expect(a.k >= 0 && a.k < GK && a.row >= 0 && a.row < GT && e.k >= 0 && e.k < GK && e.row >= 0 && e.row < GT,
                   "copy outside its stage");
            const long long atA = b * g.sA + a.at, atB = b * g.sB + e.at;
            expect(atA >= 0 && atA < extA && atB >= 0 && atB < extB, "copy outside its operand");
            if (a.valid) expect(a.at == (TA ? (long long)(kc + a.k) * g.lda + q.m0 + a.row : (long long)(q.m0 + a.row) * g.lda + kc + a.k), "wrong element of A");
            if (e.valid) expect(e.at == (TB ? (long long)(q.n0 + e.row) * g.ldb + kc + e.k : (long long)(kc + e.k) * g.ldb + q.n0 + e.row), "wrong element of B");
            expect(!a_in[a.k][a.row] && !b_in[e.k][e.row], "element copied twice");
            a_in[a.k][a.row] = b_in[e.k][e.row] = true;
          }
        for (int k = 0; k < kv; ++k)
          for (int r = 0; r < GT; ++r) expect(a_in[k][r] && b_in[k][r], "product of an element that was not copied");
        ks[bx] += kv;
      }
      // the results: two a thread (or a part of the tile for each block of a cluster)
      auto store = [&](int m, int n) {
        if (m >= g.M || n >= g.N) return;
        const long long at = (g.reduce_batch ? 0 : (long long)q.batch * g.sC) + (long long)m * g.ldc + n;
        expect(at >= 0 && at < extC, "result outside C");
        if (at >= 0 && at < extC) ++writers[at];
      };
      if (p.nslice > 1 && !p.cluster) {
        for (int tid = 0; tid < GThreads; ++tid) {
          const int m = q.m0 + tid / 8, n = q.n0 + 2 * (tid % 8);
          const long long w = ((long long)q.batch * p.nslice + by) * g.M * g.N + (long long)m * g.N + n;
          if (m < g.M && n < g.N) expect(w >= 0 && (size_t)w < work_elems, "partial sum outside the workspace");
          if (m < g.M && n + 1 < g.N) expect((size_t)(w + 1) < work_elems, "partial sum outside the workspace");
        }
      } else if (p.nslice > 1) {
        for (int tid = 0; tid < GThreads; ++tid)
          for (int e = by * GThreads + tid; e < GT * GT; e += p.nslice * GThreads) {
            const int m = q.m0 + e / GT, n = q.n0 + e % GT;
            store(m, n);
            if (g.mirror && q.n0 < q.m0) store(n, m);
          }
      } else {
        for (int tid = 0; tid < GThreads; ++tid)
          for (int x = 0; x < 2; ++x) {
            const int m = q.m0 + tid / 8, n = q.n0 + 2 * (tid % 8) + x;
            store(m, n);
            if (g.mirror && q.n0 < q.m0) store(n, m);
          }
      }
    }
  for (long long bx = 0; bx < p.ctas; ++bx)
    expect(ks[bx] == (long long)g.K * (g.reduce_batch ? g.batch : 1), "the slices do not add up to K");
  if (p.nslice <= 1 || p.cluster)
    for (int b = 0; b < nb; ++b)
      for (int m = 0; m < g.M; ++m)
        for (int n = 0; n < g.N; ++n) {
          const bool want = !g.lower_only || g.mirror || n / GT <= m / GT;
          expect(writers[b * g.sC + (long long)m * g.ldc + n] == (want ? 1 : 0), "element of C not written exactly once");
        }
}

void check(const GemmArgs& g, int sms, size_t work_elems) {
  g_now = &g;
  const GemmPlan p = gemm_plan(g, sms, work_elems);
  expect(p.chunk >= 1 && p.chunk <= GK, "chunk longer than a stage");
  expect(!p.cluster || (p.nslice >= 2 && p.nslice <= kGemmCluster), "cluster size");
  expect(p.nslice >= 1 && p.nslice <= 65535 && p.ctas >= 1 && p.ctas <= 0x7fffffffLL, "grid");
  if (g.transA && g.transB) walk<true, true>(g, p, work_elems);
  else if (g.transA) walk<true, false>(g, p, work_elems);
  else if (g.transB) walk<false, true>(g, p, work_elems);
  else walk<false, false>(g, p, work_elems);
}

}  // namespace

int main() {
  int cases = 0;
  std::map<int, int> seen;   // by kind: 0 whole, 1 cluster, 2 workspace
  auto add = [&](GemmArgs g, size_t work) {
    for (int t = 0; t < 4; ++t) {
      g.transA = t & 1;
      g.transB = t & 2;
      const int pad = cases % 3;
      g.lda = (g.transA ? g.M : g.K) + pad;
      g.ldb = (g.transB ? g.K : g.N) + pad;
      g.ldc = g.N + (g.mirror ? 0 : pad);
      g.sA = (long long)(g.transA ? g.K : g.M) * g.lda;
      g.sB = (long long)(g.transB ? g.N : g.K) * g.ldb;
      g.sC = (long long)g.M * g.ldc;
      check(g, 152, work);
      const GemmPlan p = gemm_plan(g, 152, work);
      ++seen[p.nslice == 1 ? 0 : p.cluster ? 1 : 2];
      ++cases;
    }
  };
  const int sizes[] = {1, 2, 7, 15, 16, 17, 31, 32, 33, 40, 64, 65, 100, 192, 257};
  const int ks[] = {1, 2, 8, 16, 31, 32, 33, 40, 63, 64, 65, 192, 257, 1000};
  for (int M : sizes)
    for (int N : {1, 16, 17, 40, 100, 192})
      for (int K : ks) {
        GemmArgs g;
        g.M = M; g.N = N; g.K = K;
        add(g, 1 << 22);
      }
  for (int N : sizes)   // symmetric results
    for (int K : ks)
      for (int mirror = 0; mirror < 2; ++mirror) {
        GemmArgs g;
        g.M = g.N = N; g.K = K; g.lower_only = true; g.mirror = mirror;
        add(g, 1 << 22);
      }
  for (int batch : {1, 2, 5, 38, 848})   // batches, and their sum
    for (int N : {1, 24, 40, 72})
      for (int K : {1, 5, 20, 33, 40})
        for (int red = 0; red < 2; ++red) {
          GemmArgs g;
          g.M = N; g.N = N + 3 * (1 - red); g.K = K; g.batch = batch; g.reduce_batch = red;
          g.lower_only = g.mirror = red && K % 2;
          if (g.lower_only) g.N = g.M;
          add(g, 1 << 24);
        }
  for (int K : {5000, 40000}) {   // long sums: slices through the workspace, and none where it is too small
    GemmArgs g;
    g.M = 30; g.N = 33; g.K = K;
    add(g, 1 << 22);
    add(g, 5000);
  }
  for (int k = 0; k < 3; ++k)
    if (!seen[k]) { printf("no case of kind %d\n", k); ++g_fail; }
  if (g_fail) return 1;
  printf("%d cases, OK\n", cases);
  return 0;
}
