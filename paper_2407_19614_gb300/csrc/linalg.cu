// Dense linear algebra kernels of librihf.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "../../include/rihf.h"
#include "eigh_tridiag.cuh"
#include "gemm_index.cuh"
#include "linalg.cuh"
#include "tc_gemm.cuh"

#include <mutex>
#include <unordered_map>

namespace rihf {

void raise_smem_limit(const void* kernel, int bytes) {
  static std::mutex mu;
  static std::unordered_map<const void*, int> cur;
  std::lock_guard<std::mutex> lock(mu);
  int dev = 0;
  RIHF_CUDA(cudaGetDevice(&dev));
  const void* key = (const void*)((const char*)kernel + dev);   // per device
  auto it = cur.find(key);
  if (it != cur.end() && it->second >= bytes) return;
  RIHF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  cur[key] = bytes;
}

}  // namespace rihf

namespace rihf {

static inline void count(const LaCtx& la, int n = 1) {
  if (la.launches) *la.launches += n;
}

// ------------------------------------------------------------ GEMM (FP64)

// Eight-byte asynchronous copy; zero when the element does not exist.
__device__ __forceinline__ void gemm_cp8(double* dst, const double* src, bool valid) {
  const unsigned at = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(at), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ void gemm_store(const GemmArgs& g, double* C, int m, int n, double v) {
  if (m >= g.M || n >= g.N) return;
  double* c = C + (long long)m * g.ldc + n;
  *c = g.beta == 0.0 ? g.alpha * v : g.alpha * v + g.beta * *c;
}

// grid.x: tiles x batches; grid.y: slices of the sum (K, or the batches when they
// are reduced).  Slices are summed in order: in a cluster over the slices through
// distributed shared memory (each CTA a part of the tile), or by
// splitk_reduce_kernel from `work` when there are more than a cluster holds.
// FULL: chunks of GK (K a multiple of it), whose index arithmetic needs no division.
template <bool TA, bool TB, bool FULL>
__global__ void __launch_bounds__(GThreads) dgemm_kernel(GemmArgs g, int tiles, int tn, int nslice, int kper, int bper,
                                                         int chunk_, int cluster, double* __restrict__ work) {
  const int chunk = FULL ? GK : chunk_;
  __shared__ double As[GS][GK][GT + 1], Bs[GS][GK][GT + 1];
  __shared__ double part[GT * GT];
  const int tid = threadIdx.x;
  const GemmBlock q = gemm_block(g, blockIdx.x, blockIdx.y, tiles, tn, kper, bper, chunk);
  const int batch = q.batch, slice = blockIdx.y, m0 = q.m0, n0 = q.n0, b0 = q.b0, k0 = q.k0, k1 = q.k1, per = q.per,
            total = q.total;
  auto fetch = [&](int c) {
    if (c < total) {
      const int b = b0 + c / per, kc = k0 + (c % per) * chunk;
      const double* A = g.A + (long long)b * g.sA;
      const double* B = g.B + (long long)b * g.sB;
      const int st = c % GS;
      for (int idx = tid; idx < GT * chunk; idx += GThreads) {
        const GemmElem a = gemm_elem<!TA>(idx, chunk, m0, g.M, kc, k1, g.lda), b = gemm_elem<TB>(idx, chunk, n0, g.N, kc, k1, g.ldb);
        gemm_cp8(&As[st][a.k][a.row], A + a.at, a.valid);
        gemm_cp8(&Bs[st][b.k][b.row], B + b.at, b.valid);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  const int tx = tid % 8, ty = tid / 8;   // row ty, columns 2 tx, 2 tx + 1
  double acc0 = 0.0, acc1 = 0.0;
  for (int c = 0; c < GS - 1; ++c) fetch(c);
  for (int c = 0; c < total; ++c) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(GS - 2) : "memory");
    __syncthreads();   // chunk c has arrived; the stage of chunk c - 1 is free
    fetch(c + GS - 1);
    const int st = c % GS, kc = k0 + (c % per) * chunk, kv = min(chunk, k1 - kc);
#pragma unroll 8
    for (int k = 0; k < kv; ++k) {
      const double a = As[st][k][ty];
      acc0 = fma(a, Bs[st][k][2 * tx], acc0);
      acc1 = fma(a, Bs[st][k][2 * tx + 1], acc1);
    }
  }
  if (nslice > 1 && !cluster) {
    const long long slot = (long long)batch * nslice + slice;
    const int m = m0 + ty, n = n0 + 2 * tx;
    double* w = work + slot * g.M * g.N + (long long)m * g.N + n;
    if (m < g.M && n < g.N) w[0] = acc0;
    if (m < g.M && n + 1 < g.N) w[1] = acc1;
    return;
  }
  double* C = g.C + (g.reduce_batch ? 0 : (long long)batch * g.sC);
  if (nslice > 1) {
    namespace cg = cooperative_groups;
    auto cl = cg::this_cluster();
    part[ty * GT + 2 * tx] = acc0;
    part[ty * GT + 2 * tx + 1] = acc1;
    cl.sync();
    for (int e = slice * GThreads + tid; e < GT * GT; e += nslice * GThreads) {
      double s = 0.0;
      for (int q = 0; q < nslice; ++q) s += *cl.map_shared_rank(part + e, q);
      const int m = m0 + e / GT, n = n0 + e % GT;
      gemm_store(g, C, m, n, s);
      if (g.mirror && n0 < m0) gemm_store(g, C, n, m, s);
    }
    cl.sync();   // no CTA leaves while its partial tile is read
    return;
  }
  const int m = m0 + ty, n = n0 + 2 * tx;
  gemm_store(g, C, m, n, acc0);
  gemm_store(g, C, m, n + 1, acc1);
  if (g.mirror && n0 < m0) {
    gemm_store(g, C, n, m, acc0);
    gemm_store(g, C, n + 1, m, acc1);
  }
}

__global__ void splitk_reduce_kernel(GemmArgs g, int nsplit, const double* __restrict__ work) {
  long long total = (long long)g.M * g.N * (g.reduce_batch ? 1 : g.batch);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    long long mn = idx % ((long long)g.M * g.N);
    int b = (int)(idx / ((long long)g.M * g.N));
    int m = (int)(mn / g.N), n = (int)(mn % g.N);
    if (g.lower_only && (n / GT) > (m / GT)) continue;
    double s = 0.0;
    for (int q = 0; q < nsplit; ++q) s += work[((long long)b * nsplit + q) * g.M * g.N + mn];
    double* C = g.C + (g.reduce_batch ? 0 : (long long)b * g.sC);
    gemm_store(g, C, m, n, s);
    if (g.mirror && (n / GT) < (m / GT)) gemm_store(g, C, n, m, s);
  }
}

// The tensor-core route of dgemm (see LaCtx::tcA): op(A) as rows M, K and
// op(B)^T as rows N, K, both sliced into 7 digits; C stored (beta 0) or
// accumulated (beta 1).  Returns false when the product does not qualify.
static bool dgemm_tc(const LaCtx& la, const GemmArgs& g) {
  if (!la.tcA || !la.tcB || g.batch != 1 || g.reduce_batch ||
      !(g.beta == 0.0 || g.beta == 1.0) || g.K <= 0)
    return false;
  if ((double)g.M * g.N * g.K < la.tc_min_work) return false;
  if ((g.K + kOzChunk - 1) / kOzChunk > kOzMaxChunksPerBlock) return false;
  auto fits = [](const OzBuf* b, int rows, int K) {
    return oz_plane_elems(rows, K, kOzMaxDigits) <= b->cap &&
           (size_t)((rows + kOzTileM - 1) / kOzTileM * kOzTileM) <= b->ecap;
  };
  if (!fits(la.tcA, g.M, g.K) || !fits(la.tcB, g.N, g.K)) return false;
  // element (m, k) of op(A) and (n, k) of op(B)^T
  OzGemmArgs o;
  o.A = oz_slice(la, g.A, g.M, g.K, g.transA ? 1 : g.lda, g.transA ? g.lda : 1, 0, g.K, kOzMaxDigits, 0, *la.tcA);
  o.B = oz_slice(la, g.B, g.N, g.K, g.transB ? g.ldb : 1, g.transB ? 1 : g.ldb, 0, g.K, kOzMaxDigits, 0, *la.tcB);
  o.M = g.M; o.N = g.N; o.s = kOzMaxDigits; o.alpha = g.alpha; o.C = g.C; o.cs_m1 = g.ldc; o.cs_n = 1;
  o.accumulate = g.beta == 1.0;
  o.lower_only = g.lower_only;
  oz_gemm(la, o);
  return true;
}

void dgemm(const LaCtx& la, const GemmArgs& g) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return;
  if (dgemm_tc(la, g)) {
    if (g.mirror) symmetrize_lower(la, g.C, g.N, 1);
    return;
  }
  const GemmPlan p = gemm_plan(g, la.sms, la.work_elems);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr{};
  cfg.gridDim = dim3((unsigned)p.ctas, (unsigned)p.nslice, 1);
  cfg.blockDim = dim3(GThreads, 1, 1);
  cfg.stream = la.stream;
  if (p.cluster) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = (unsigned)p.nslice;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
  auto run = [&](auto kernel) {
    RIHF_CUDA(cudaLaunchKernelEx(&cfg, kernel, g, p.tiles, p.tn, p.nslice, p.kper, p.bper, p.chunk, p.cluster, la.work));
  };
  auto pick = [&](auto full) {
    constexpr bool F = decltype(full)::value;
    if (g.transA && g.transB) run(dgemm_kernel<true, true, F>);
    else if (g.transA) run(dgemm_kernel<true, false, F>);
    else if (g.transB) run(dgemm_kernel<false, true, F>);
    else run(dgemm_kernel<false, false, F>);
  };
  if (p.chunk == GK) pick(std::true_type());
  else pick(std::false_type());
  count(la);
  if (p.nslice > 1 && !p.cluster) {
    const long long total = (long long)g.M * g.N * (g.reduce_batch ? 1 : g.batch);
    const int blocks = (int)std::min<long long>((total + 255) / 256, 8LL * la.sms);
    splitk_reduce_kernel<<<blocks, 256, 0, la.stream>>>(g, p.nslice, la.work);
    RIHF_LAUNCH_CHECK();
    count(la);
  }
}

__global__ void symmetrize_lower_kernel(double* X, int n) {
  __shared__ double t[32][33];
  int bi = blockIdx.y, bj = blockIdx.x;   // destination tile (bi, bj) with bi <= bj (upper)
  if (bi > bj) return;
  double* S = X + (size_t)blockIdx.z * n * n;
  // source tile (bj, bi) in the lower triangle
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int i = bj * 32 + r, j = bi * 32 + threadIdx.x;
    t[r][threadIdx.x] = (i < n && j < n) ? S[(size_t)i * n + j] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int i = bi * 32 + r, j = bj * 32 + threadIdx.x;   // upper element (i, j), j > i
    if (i < n && j < n && j > i) S[(size_t)i * n + j] = t[threadIdx.x][r];
  }
}

void symmetrize_lower(const LaCtx& la, double* X, int n, int batch) {
  int nt = ceil_div(n, 32);
  symmetrize_lower_kernel<<<dim3(nt, nt, batch), dim3(32, 8), 0, la.stream>>>(X, n);
  RIHF_LAUNCH_CHECK();
  count(la);
}

// ------------------------------------------------------------ Cholesky

constexpr int CB = 32;

// One step of the right-looking blocked Cholesky (block CB = 32), in one launch
// of 128-thread blocks.  Every block factors the diagonal block L_kk itself
// (the same instructions on the same data, so every block gets the same bits):
// lane r holds row r, warp w the columns c = 4 t + w, and each pivot column is
// broadcast through shared memory, so the narrow FP64 pipes of all four SM
// sub-partitions share the rank-1 updates while one warp runs the pivot's
// reciprocal square root.  Block 0 stores L_kk in Ld (the diagonal block of A
// is still being read by the other blocks; chol_finish_kernel copies it in).
// Then the panel rows r >= k + b solve y L_kk^T = a_r by forward substitution,
// eight lanes a row as in trsv_lanes_kernel.  (Four lanes a row, each entry a dot
// product reduced by shuffles, made the rows 2/3 of the step's 34 us.)
__global__ void __launch_bounds__(128) chol_step_kernel(double* A, int n, int k, int b, int* flag, double* Ld) {
  __shared__ double l[CB][CB + 1];
  __shared__ double piv[2][CB];
  __shared__ double rd[CB];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double a[CB / 4];
#pragma unroll
  for (int t = 0; t < CB / 4; ++t) {
    const int c = 4 * t + w;
    a[t] = (lane < b && c < b && c <= lane) ? A[(size_t)(k + lane) * n + k + c] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < CB; ++j) {
    if (j < b) {
      if (w == (j & 3)) {
        double d = __shfl_sync(0xffffffffu, a[j >> 2], j);
        if (!(d > 0.0)) {
          if (lane == 0 && blockIdx.x == 0) atomicExch(flag, 1);
          d = 1.0;
          if (lane == j) a[j >> 2] = 1.0;
        }
        // rows above the pivot hold zeros and row j holds d itself, so one
        // multiply gives l_jj = d r and the column below scaled by r
        a[j >> 2] *= rsqrt(d);
        piv[j & 1][lane] = a[j >> 2];
      }
      __syncthreads();   // also orders the reuse of piv[j & 1] two steps on
      const double lj = piv[j & 1][lane];
#pragma unroll
      for (int t = 0; t < CB / 4; ++t) {
        const int c = 4 * t + w;
        if (c > j && lane >= c) a[t] = fma(-lj, piv[j & 1][c], a[t]);
      }
    }
  }
#pragma unroll
  for (int t = 0; t < CB / 4; ++t) {
    const int c = 4 * t + w;
    l[lane][c] = a[t];
    if (blockIdx.x == 0 && lane < b && c < b) Ld[(size_t)(k + lane) * CB + c] = a[t];
  }
  __syncthreads();
  if (threadIdx.x < CB) {
    rd[threadIdx.x] = threadIdx.x < b ? 1.0 / l[threadIdx.x][threadIdx.x] : 0.0;
    l[threadIdx.x][threadIdx.x] = 0.0;   // entries that are done subtract zero
  }
  __syncthreads();
  const int s = lane & 7;
  for (int r0 = k + b + (blockIdx.x * 4 + w) * 4; r0 < n; r0 += gridDim.x * 16) {
    const int r = r0 + (lane >> 3);
    double y[CB / 8];
#pragma unroll
    for (int q = 0; q < CB / 8; ++q) y[q] = r < n && s + 8 * q < b ? A[(size_t)r * n + k + s + 8 * q] : 0.0;
#pragma unroll
    for (int i = 0; i < CB; ++i) {
      const double v = __shfl_sync(0xffffffffu, y[i / 8] * rd[i], i & 7, 8);
      if (s == (i & 7)) y[i / 8] = v;
#pragma unroll
      for (int q = i / 8; q < CB / 8; ++q) y[q] = fma(-l[s + 8 * q][i], v, y[q]);
    }
#pragma unroll
    for (int q = 0; q < CB / 8; ++q)
      if (r < n && s + 8 * q < b) A[(size_t)r * n + k + s + 8 * q] = y[q];
  }
}

// The diagonal blocks from Ld into A; the upper triangle zeroed.
__global__ void chol_finish_kernel(double* A, int n, const double* __restrict__ Ld) {
  long long total = (long long)n * n;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / n), j = (int)(idx % n);
    if (j > i) A[idx] = 0.0;
    else if (i / CB == j / CB) A[idx] = Ld[(size_t)i * CB + (j % CB)];
  }
}

void cholesky(const LaCtx& la, double* A, int n, double* scratch) {
  double* Ld = scratch;   // n x CB: the factored diagonal blocks
  for (int k = 0; k < n; k += CB) {
    int b = std::min(CB, n - k);
    int rest = n - k - b;
    // L_kk, and A[k+b:, k:k+b] <- A[k+b:, k:k+b] L_kk^{-T}
    const int blocks = std::max(1, std::min(ceil_div(rest, 16), la.sms));
    chol_step_kernel<<<blocks, 128, 0, la.stream>>>(A, n, k, b, la.flag, Ld);
    RIHF_LAUNCH_CHECK();
    count(la);
    if (rest <= 0) break;
    // trailing update: A[k+b:, k+b:] -= panel panel^T, lower tiles only (the
    // factorisation never reads the upper triangle; it is zeroed at the end)
    GemmArgs u;
    u.M = rest; u.N = rest; u.K = b;
    u.A = A + (size_t)(k + b) * n + k; u.lda = n;
    u.B = A + (size_t)(k + b) * n + k; u.ldb = n; u.transB = true;
    u.C = A + (size_t)(k + b) * n + k + b; u.ldc = n;
    u.alpha = -1.0; u.beta = 1.0;
    u.lower_only = true;
    dgemm(la, u);
  }
  chol_finish_kernel<<<std::max(1, std::min(ceil_div((long long)n * n, 256), 8 * la.sms)), 256, 0, la.stream>>>(
      A, n, Ld);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void identity_kernel(double* X, int n) {
  long long total = (long long)n * n;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x)
    X[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

void identity(const LaCtx& la, double* X, int n) {
  identity_kernel<<<std::max(1, std::min(ceil_div((long long)n * n, 256), 8 * la.sms)), 256, 0, la.stream>>>(X, n);
  RIHF_LAUNCH_CHECK();
  count(la);
}

// Substitution inside one diagonal block: every thread owns one column j of the
// b x ncol slab X[k:k+b, :] and solves L_kk y = x (trans = 0) or L_kk^T y = x
// (trans = 1) in registers; L_kk is staged in shared memory.  Substitution (not
// a product with an explicit block inverse) keeps the accuracy of the classical
// algorithm when the auxiliary functions of one atom make L_kk ill-conditioned.
__global__ void __launch_bounds__(256) trsv_block_kernel(const double* __restrict__ L, int n, int k, int b,
                                                         double* __restrict__ X, long long ncol, int trans,
                                                         int symcols) {
  __shared__ double l[CB][CB + 1];
  __shared__ double rd[CB];
  for (int i = threadIdx.x; i < CB * CB; i += blockDim.x) {
    int r = i / CB, c = i % CB;
    l[r][c] = (r < b && c < b) ? L[(size_t)(k + r) * n + k + c] : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < CB; i += blockDim.x) rd[i] = i < b ? 1.0 / l[i][i] : 0.0;
  __syncthreads();
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < ncol; j += (long long)gridDim.x * blockDim.x) {
    if (symcols > 0 && (j % symcols) > (j / symcols)) continue;   // strict upper triangle: never used
    double y[CB];
#pragma unroll
    for (int i = 0; i < CB; ++i) y[i] = i < b ? X[(size_t)(k + i) * ncol + j] : 0.0;
    if (!trans) {
#pragma unroll
      for (int i = 0; i < CB; ++i) {
        if (i >= b) break;
        double s = y[i];
#pragma unroll
        for (int q = 0; q < i; ++q) s -= l[i][q] * y[q];
        y[i] = s * rd[i];
      }
    } else {
#pragma unroll
      for (int i = CB - 1; i >= 0; --i) {
        if (i >= b) continue;
        double s = y[i];
#pragma unroll
        for (int q = i + 1; q < CB; ++q)
          if (q < b) s -= l[q][i] * y[q];
        y[i] = s * rd[i];
      }
    }
#pragma unroll
    for (int i = 0; i < CB; ++i)
      if (i < b) X[(size_t)(k + i) * ncol + j] = y[i];
  }
}

// The same with eight lanes a column: lane s holds rows s, s + 8, s + 16, s + 24, and
// each solved entry is passed round by a shuffle.  A column's chain is then about
// five FP64 instructions an entry instead of up to 32 (10 k clocks instead of 34 k),
// for 1.6 times the FP64 instructions: faster while the columns leave the SMs short
// of warps.  The diagonal of l is zero (it is in rd), so rows that are done subtract
// zero times the entry.
__global__ void __launch_bounds__(128) trsv_lanes_kernel(const double* __restrict__ L, int n, int k, int b,
                                                         double* __restrict__ X, long long ncol, int trans) {
  __shared__ double l[CB][CB + 1];
  __shared__ double rd[CB];
  for (int i = threadIdx.x; i < CB * CB; i += 128) {
    const int r = i / CB, c = i % CB;
    const double v = r < b && c <= r ? L[(size_t)(k + r) * n + k + c] : 0.0;
    if (r == c) rd[r] = r < b ? 1.0 / v : 0.0;
    // trans: the columns of L are walked, so the transpose is kept
    if (trans) l[c][r] = r == c ? 0.0 : v;
    else l[r][c] = r == c ? 0.0 : v;
  }
  __syncthreads();
  const int s = threadIdx.x & 7;
  const long long j = blockIdx.x * 16LL + (threadIdx.x >> 3);
  double y[CB / 8];
#pragma unroll
  for (int q = 0; q < CB / 8; ++q) {
    const int r = s + 8 * q;
    y[q] = r < b && j < ncol ? X[(size_t)(k + r) * ncol + j] : 0.0;
  }
  if (!trans) {
#pragma unroll
    for (int i = 0; i < CB; ++i) {
      const double v = __shfl_sync(0xffffffffu, y[i / 8] * rd[i], i & 7, 8);
      if (s == (i & 7)) y[i / 8] = v;
#pragma unroll
      for (int q = i / 8; q < CB / 8; ++q) y[q] = fma(-l[s + 8 * q][i], v, y[q]);
    }
  } else {
#pragma unroll
    for (int i = CB - 1; i >= 0; --i) {
      const double v = __shfl_sync(0xffffffffu, y[i / 8] * rd[i], i & 7, 8);
      if (s == (i & 7)) y[i / 8] = v;
#pragma unroll
      for (int q = 0; q <= i / 8; ++q) y[q] = fma(-l[s + 8 * q][i], v, y[q]);
    }
  }
  if (j < ncol)
#pragma unroll
    for (int q = 0; q < CB / 8; ++q) {
      const int r = s + 8 * q;
      if (r < b) X[(size_t)(k + r) * ncol + j] = y[q];
    }
}

// One diagonal block of a solve.  Eight lanes a column up to 64 columns an SM (about
// 9700, where they come to four warps per SM sub-partition: 29 k clocks of FP64
// instructions against the 34 k of one column's chain in one thread), one thread a
// column above; narrow blocks then spread few columns over many SMs.
static void trsv_block(const LaCtx& la, const double* L, int n, int k, int b, double* X, long long ncol, bool trans,
                       int symcols) {
  if (ncol <= 64LL * la.sms) {
    trsv_lanes_kernel<<<(unsigned)((ncol + 15) / 16), 128, 0, la.stream>>>(L, n, k, b, X, ncol, trans ? 1 : 0);
  } else {
    const long long per = (ncol + 2LL * la.sms - 1) / (2LL * la.sms);   // columns per block for two blocks per SM
    const int threads = (int)std::min<long long>(256, std::max<long long>(32, (per + 31) / 32 * 32));
    const int blocks = (int)std::max<long long>(1, std::min<long long>((ncol + threads - 1) / threads, 16LL * la.sms));
    trsv_block_kernel<<<blocks, threads, 0, la.stream>>>(L, n, k, b, X, ncol, trans ? 1 : 0, symcols);
  }
  RIHF_LAUNCH_CHECK();
  count(la);
}

void trsm_lower(const LaCtx& la, const double* L, int n, double* X, long long ncol, bool trans, int symcols,
                double* tmp) {
  (void)tmp;
  const int nb = ceil_div(n, CB);
  for (int q = 0; q < nb; ++q) {
    const int kb = trans ? nb - 1 - q : q;
    const int k = kb * CB, b = std::min(CB, n - k);
    trsv_block(la, L, n, k, b, X, ncol, trans, symcols);
    GemmArgs u;
    u.N = (int)ncol; u.K = b;
    u.B = X + (size_t)k * ncol; u.ldb = (int)ncol;
    u.alpha = -1.0; u.beta = 1.0;
    if (!trans) {
      // X[k+b:, :] -= L[k+b:, k:k+b] X_k
      u.M = n - k - b;
      u.A = L + (size_t)(k + b) * n + k; u.lda = n;
      u.C = X + (size_t)(k + b) * ncol; u.ldc = (int)ncol;
    } else {
      // X[0:k, :] -= L[k:k+b, 0:k]^T X_k
      u.M = k;
      u.A = L + (size_t)k * n; u.lda = n; u.transA = true;
      u.C = X; u.ldc = (int)ncol;
    }
    if (u.M > 0) dgemm(la, u);
  }
}

void trsm_lower_tc(const LaCtx& la, const double* L, int n, double* X, long long ncol, int symcols,
                   const TrsmTcScratch& sc) {
  constexpr int PB = kTrsmPanel;   // inner panel width (K of the inner digit-plane updates)
  // X[r0 + M rows] -= L[r0.., k..k+kk) X[k..k+kk) on the tensor cores
  auto tc_update = [&](int r0, int M, int k, int kk) {
    if (M <= 0) return;
    OzGemmArgs g;
    g.A = oz_slice(la, L + (size_t)r0 * n + k, M, kk, n, 1, 0, kk, kOzMaxDigits, 0, sc.L);
    g.B = oz_slice(la, X + (size_t)k * ncol, (int)ncol, kk, 1, ncol, 0, kk, kOzMaxDigits, 0, sc.X);
    g.M = M; g.N = (int)ncol; g.s = kOzMaxDigits; g.alpha = -1.0;
    g.C = X + (size_t)r0 * ncol; g.cs_m1 = ncol; g.cs_n = 1;
    g.accumulate = true; g.symcols = symcols;
    oz_gemm(la, g);
  };
  for (int ko = 0; ko < n; ko += kTrsmOuter) {
  const int ke = std::min(n, ko + kTrsmOuter);
  for (int k = ko; k < ke; k += PB) {
    const int pb = std::min(PB, ke - k);
    // the panel in FP64: 32-row substitution blocks and their in-panel updates
    for (int k2 = k; k2 < k + pb; k2 += CB) {
      const int b = std::min(CB, k + pb - k2);
      trsv_block(la, L, n, k2, b, X, ncol, false, symcols);
      const int m2 = k + pb - (k2 + b);
      if (m2 > 0) {
        GemmArgs u;
        u.M = m2; u.N = (int)ncol; u.K = b;
        u.A = L + (size_t)(k2 + b) * n + k2; u.lda = n;
        u.B = X + (size_t)k2 * ncol; u.ldb = (int)ncol;
        u.C = X + (size_t)(k2 + b) * ncol; u.ldc = (int)ncol;
        u.alpha = -1.0; u.beta = 1.0;
        dgemm(la, u);
      }
    }
    // rows of the outer panel below this panel
    tc_update(k + pb, ke - k - pb, k, pb);
  }
  // all rows below the outer panel: one rank-(ke - ko) update
  tc_update(ke, n - ke, ko, ke - ko);
  }
}

void trsm_lower_t_tc(const LaCtx& la, const double* L, int n, double* X, long long ncol, int symcols,
                     const TrsmTcScratch& sc) {
  constexpr int PB = kTrsmPanel;
  // X[r0 .. r0+M) -= L[k..k+kk, r0..r0+M)^T X[k..k+kk) on the tensor cores
  auto tc_update = [&](int r0, int M, int k, int kk) {
    if (M <= 0) return;
    OzGemmArgs g;
    g.A = oz_slice(la, L + (size_t)k * n + r0, M, kk, 1, n, 0, kk, kOzMaxDigits, 0, sc.L);
    g.B = oz_slice(la, X + (size_t)k * ncol, (int)ncol, kk, 1, ncol, 0, kk, kOzMaxDigits, 0, sc.X);
    g.M = M; g.N = (int)ncol; g.s = kOzMaxDigits; g.alpha = -1.0;
    g.C = X + (size_t)r0 * ncol; g.cs_m1 = ncol; g.cs_n = 1;
    g.accumulate = true; g.symcols = symcols;
    oz_gemm(la, g);
  };
  // outer panels [ko, ke) from the bottom; inner 64-row panels and 32-row
  // substitution blocks aligned to multiples of their size, also from the bottom
  for (int ko = (n - 1) / kTrsmOuter * kTrsmOuter; ko >= 0; ko -= kTrsmOuter) {
    const int ke = std::min(n, ko + kTrsmOuter);
    for (int k = ko + (ke - ko - 1) / PB * PB; k >= ko; k -= PB) {
      const int kend = std::min(ke, k + PB);
      for (int k2 = k + (kend - k - 1) / CB * CB; k2 >= k; k2 -= CB) {
        const int b = std::min(CB, kend - k2);
        trsv_block(la, L, n, k2, b, X, ncol, true, symcols);
        if (k2 > k) {   // rows [k, k2) of the panel: X -= L[k2:k2+b, k:k2]^T X_k2
          GemmArgs u;
          u.M = k2 - k; u.N = (int)ncol; u.K = b;
          u.A = L + (size_t)k2 * n + k; u.lda = n; u.transA = true;
          u.B = X + (size_t)k2 * ncol; u.ldb = (int)ncol;
          u.C = X + (size_t)k * ncol; u.ldc = (int)ncol;
          u.alpha = -1.0; u.beta = 1.0;
          dgemm(la, u);
        }
      }
      // rows of the outer panel above this panel
      tc_update(ko, k - ko, k, kend - k);
    }
    // all rows above the outer panel: one rank-(ke - ko) update
    tc_update(0, ko, ko, ke - ko);
  }
}

// ------------------------------------------------------------ eigensolver

// One-sided (Hestenes) Jacobi in FP32: with B = A + sigma I positive definite
// (sigma from a Gershgorin bound), column rotations U <- U J drive the columns of
// U = B V to mutual orthogonality; then v_j = u_j / |u_j| and lambda_j = |u_j| -
// sigma.  Only U (n x n, column-major) is stored.  A is scaled by the power of two
// that brings its largest row sum into [1, 2) (which changes no rounding): unscaled,
// the fourth powers of the entries that the convergence test multiplies leave the FP32
// range at norms below 1e-10 and above 1e10.
//
// The columns form nb blocks of H (nb even); in a round a warp holds the two
// blocks of one block pair in registers (R rows of every column per lane) and
// rotates every column pair across them (round 0 also the pairs inside each
// block); a sweep is the nb - 1 rounds of the round-robin order.  Squared column
// norms are carried by the rotation identities |u_p'|^2 = |u_p|^2 - t (u_p . u_q),
// |u_q'|^2 = |u_q|^2 + t (u_p . u_q) and recomputed at every sweep, so a pair costs
// one reduction.  The H rotations of one step are independent and written without
// branches, so that their reductions overlap.
//
// What bounds it is the latency of a round, so that a single CTA with all 32 warps
// of a 192 x 192 problem on one SM was bound by that SM's issue slots and shared
// memory (0.45 ms a sweep).  Above n = 64 the pairs are spread over a cluster of
// CL = 8 CTAs, the columns pass through L2 (.cg loads and stores) and a cluster
// barrier ends each round: 0.24 ms a sweep.  Up to n = 64 one CTA with U in shared
// memory is faster than the barrier (n = 24: 81 us to convergence, 104 us when its
// rounds ran over 64 mostly empty blocks).
constexpr int kJacobiCluster = 8;
constexpr int kJacobiSmall = 64;

template <int H, int R, int CL>
__global__ void __launch_bounds__(CL == 1 ? 1024 : 32 * 4)
    jacobi1s_kernel(const double* __restrict__ A, int n, int m, float* gU, float* __restrict__ V, float* W, int nb,
                    int max_sweeps, float tol) {
  namespace cg = cooperative_groups;
  extern __shared__ float sm[];
  __shared__ float red[33];
  __shared__ int flag;   // a pair was rotated in this sweep
  const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CL == 1 ? 0 : (int)blockIdx.x, gw = rank * warps + warp, nw = CL * warps;   // warp of the cluster
  float* U = CL == 1 ? sm : gU;
  auto sync = [&]() {
    if constexpr (CL == 1) __syncthreads();
    else cg::this_cluster().sync();
  };
  auto ld = [&](const float* x) -> float { return CL == 1 ? *x : __ldcg(x); };
  auto st = [&](float* x, float v) {
    if constexpr (CL == 1) *x = v;
    else __stcg(x, v);
  };
  const float tol2 = tol * tol;
  // sigma = 1.05 max_i sum_j |A_ij|
  float g = 0.f;
  for (int i = gw; i < n; i += nw) {
    float s = 0.f;
    for (int j = lane; j < n; j += 32) s += fabsf((float)A[(size_t)i * n + j]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    g = fmaxf(g, s);
  }
  if (lane == 0) red[warp] = g;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < warps; ++w) t = fmaxf(t, red[w]);
    red[32] = t;
  }
  sync();
  float top = red[32];
  if constexpr (CL > 1)
    for (int q = 0; q < CL; ++q) top = fmaxf(top, *cg::this_cluster().map_shared_rank(red + 32, q));
  const int ex = min(max((__float_as_int(top) >> 23) - 127, -126), 126);   // top >= 0
  const float down = __int_as_float((127 - ex) << 23), up = __int_as_float((127 + ex) << 23);   // 2^-ex, 2^ex
  const float sigma = 1.05f * (top * down) + 1e-20f;
  for (int j = gw; j < n; j += nw)
    for (int i = lane; i < n; i += 32)
      st(U + (size_t)j * n + i, (float)A[(size_t)i * n + j] * down + (i == j ? sigma : 0.f));
  sync();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (threadIdx.x == 0) flag = 0;
    // squared norms, kept in W until the end
    for (int j = gw; j < n; j += nw) {
      const float* u = U + (size_t)j * n;
      float s2 = 0.f;
      for (int i = lane; i < n; i += 32) {
        const float x = ld(u + i);
        s2 = fmaf(x, x, s2);
      }
      for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      if (lane == 0) __stcg(W + j, s2);
    }
    sync();
    bool rotated = false;
    for (int r = 0; r < nb - 1; ++r) {
      if (gw < nb / 2) {
        const int bA = gw == 0 ? nb - 1 : (r + gw) % (nb - 1), bB = gw == 0 ? r : (r - gw + nb - 1) % (nb - 1);
        float x[2 * H][R], cn[2 * H];
#pragma unroll
        for (int c = 0; c < 2 * H; ++c) {
          const int col = c < H ? bA * H + c : bB * H + c - H;
          cn[c] = col < n ? __ldcg(W + col) : 0.f;
#pragma unroll
          for (int e = 0; e < R; ++e) {
            const int i = lane + 32 * e;
            x[c][e] = col < n && i < n ? ld(U + (size_t)col * n + i) : 0.f;
          }
        }
        auto rot = [&](float (&xp)[R], float (&xq)[R], float& a, float& b) {
          float c = 0.f;
#pragma unroll
          for (int e = 0; e < R; ++e) c = fmaf(xp[e], xq[e], c);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
          // fast divisions and roots: the angle needs a few digits only, and c^2 + s^2 = 1
          // holds to the rounding of rsqrtf
          const bool act = c * c > (tol2 * a) * b;   // not a converged pair, nor a zero (padding) column
          rotated |= act;
          const float zeta = fminf(fmaxf(__fdividef(b - a, 2.f * (act ? c : 1.f)), -1e18f), 1e18f);
          const float z2 = fmaf(zeta, zeta, 1.f);
          const float t = act ? copysignf(__fdividef(1.f, fabsf(zeta) + z2 * rsqrtf(z2)), zeta) : 0.f;
          const float cs = act ? rsqrtf(fmaf(t, t, 1.f)) : 1.f, sn = cs * t;
#pragma unroll
          for (int e = 0; e < R; ++e) {
            const float u = xp[e], v = xq[e];
            xp[e] = cs * u - sn * v;
            xq[e] = sn * u + cs * v;
          }
          a -= t * c;
          b += t * c;
        };
        if (r == 0) {
#pragma unroll
          for (int p = 0; p < H; ++p)
#pragma unroll
            for (int q = p + 1; q < H; ++q) {
              rot(x[p], x[q], cn[p], cn[q]);
              rot(x[H + p], x[H + q], cn[H + p], cn[H + q]);
            }
        }
#pragma unroll
        for (int d = 0; d < H; ++d)
#pragma unroll
          for (int p = 0; p < H; ++p) rot(x[p], x[H + (p + d) % H], cn[p], cn[H + (p + d) % H]);
#pragma unroll
        for (int c = 0; c < 2 * H; ++c) {
          const int col = c < H ? bA * H + c : bB * H + c - H;
          if (col < n) {
#pragma unroll
            for (int e = 0; e < R; ++e) {
              const int i = lane + 32 * e;
              if (i < n) st(U + (size_t)col * n + i, x[c][e]);
            }
            if (lane == 0) __stcg(W + col, cn[c]);
          }
        }
      }
      sync();
    }
    if (rotated && lane == 0) flag = 1;
    sync();
    bool more = flag != 0;
    if constexpr (CL > 1)
      for (int q = 0; q < CL; ++q) more |= *cg::this_cluster().map_shared_rank(&flag, q) != 0;
    sync();   // every flag has been read
    if (!more) break;
  }
  // eigenpairs of the orthogonalised columns; V row-major n x m
  for (int j = gw; j < n; j += nw) {
    const float* u = U + (size_t)j * n;
    float s = 0.f;
    for (int i = lane; i < n; i += 32) {
      const float x = ld(u + i);
      s = fmaf(x, x, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float nrm = sqrtf(s), inv = nrm > 0.f ? 1.f / nrm : 0.f;
    for (int i = lane; i < n; i += 32) V[(size_t)i * m + j] = ld(u + i) * inv;
    if (lane == 0) W[j] = (nrm - sigma) * up;
  }
}

static void jacobi(const LaCtx& la, const double* A, int n, int m, float* gU, float* V, float* W, int max_sweeps,
                   float tol) {
  const bool small = n <= kJacobiSmall;
  const int H = small ? 1 : 4, nb = std::max(2, (ceil_div(n, H) + 1) / 2 * 2);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr{};
  cfg.stream = la.stream;
  if (small) {
    cfg.gridDim = dim3(1, 1, 1);
    cfg.blockDim = dim3(32 * nb / 2, 1, 1);
    cfg.dynamicSmemBytes = (size_t)n * n * sizeof(float);
    RIHF_CUDA(cudaLaunchKernelEx(&cfg, jacobi1s_kernel<1, 2, 1>, A, n, m, gU, V, W, nb, max_sweeps, tol));
  } else {
    cfg.gridDim = dim3(kJacobiCluster, 1, 1);
    cfg.blockDim = dim3(32 * ceil_div(nb / 2, kJacobiCluster), 1, 1);
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kJacobiCluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    auto run = [&](auto kernel) { RIHF_CUDA(cudaLaunchKernelEx(&cfg, kernel, A, n, m, gU, V, W, nb, max_sweeps, tol)); };
    if (n <= 128) run(jacobi1s_kernel<4, 4, kJacobiCluster>);
    else if (n <= 192) run(jacobi1s_kernel<4, 6, kJacobiCluster>);
    else run(jacobi1s_kernel<4, 8, kJacobiCluster>);
  }
  count(la);
}

// Sort eigenpairs ascending (rank sort) and expand to FP64: X[:, rank] = V[:, i].
__global__ void eig_sort_kernel(const float* __restrict__ V, const float* __restrict__ W, int n, int m, double* X,
                                double* Wd) {
  __shared__ int rank[kEighMax];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    float wi = W[i];
    int r = 0;
    for (int j = 0; j < n; ++j) {
      float wj = W[j];
      if (wj < wi || (wj == wi && j < i)) ++r;
    }
    rank[i] = r;
  }
  __syncthreads();
  // every block ranks all n values, then moves its own rows
  for (int row = blockIdx.x; row < n; row += gridDim.x)
    for (int i = threadIdx.x; i < n; i += blockDim.x) X[(size_t)row * n + rank[i]] = (double)V[row * m + i];
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n; i += blockDim.x) Wd[rank[i]] = (double)W[i];
}

// Ogita-Aishima step pieces: lam_i = S_ii/(1-R_ii); E_ij as in their Algorithm 1.
__global__ void oa_lambda_kernel(const double* R, const double* S, int n, double* lam) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    lam[i] = S[(size_t)i * n + i] / (1.0 - R[(size_t)i * n + i]);
}

// Partial sums of ||S - diag(lam)||_F^2, ||R||_F^2 and ||A||_F^2, block b into
// part[3b .. 3b+2] (oa_e_kernel folds them in a fixed order).
constexpr int kOaParts = 64;
__global__ void oa_norms_kernel(const double* R, const double* S, const double* A, const double* lam, int n,
                                double* part) {
  __shared__ double r0[32], r1[32], r2[32];
  double a0 = 0, a1 = 0, a2 = 0;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * n;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / n), j = (int)(idx % n);
    double s = S[idx] - (i == j ? lam[i] : 0.0);
    a0 += s * s;
    a1 += R[idx] * R[idx];
    a2 += A[idx] * A[idx];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    a2 += __shfl_xor_sync(0xffffffffu, a2, o);
  }
  if ((threadIdx.x & 31) == 0) { r0[threadIdx.x / 32] = a0; r1[threadIdx.x / 32] = a1; r2[threadIdx.x / 32] = a2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0, s1 = 0, s2 = 0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) { s0 += r0[w]; s1 += r1[w]; s2 += r2[w]; }
    part[3 * blockIdx.x] = s0; part[3 * blockIdx.x + 1] = s1; part[3 * blockIdx.x + 2] = s2;
  }
}

__global__ void oa_e_kernel(const double* R, const double* S, const double* lam, const double* part, int nparts,
                            int n, double* E) {
  __shared__ double sh_delta, sh_min;
  if (threadIdx.x < 32) {   // fold the partial sums (fixed order: deterministic)
    double s0 = 0, s1 = 0, s2 = 0;
    for (int b = threadIdx.x; b < nparts; b += 32) {
      s0 += part[3 * b];
      s1 += part[3 * b + 1];
      s2 += part[3 * b + 2];
    }
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (threadIdx.x == 0) {
      sh_delta = 2.0 * (sqrt(s0) + sqrt(s2) * sqrt(s1));
      sh_min = 1e-14 * sqrt(s2);
    }
  }
  __syncthreads();
  const double delta = sh_delta, dmin = sh_min;
  // A pair is rotated when its gap exceeds the global cluster threshold (as in
  // the method), or when its own first-order correction is small, |E_ij| < 1/8.
  // The threshold bounds the spectral norms of the residuals by their
  // Frobenius norms, which for large n exceed them by up to sqrt(n): pairs far
  // apart relative to their own coupling would otherwise count as clustered and
  // never rotate (at n = 1856 the refinement then stalls near FP32 accuracy).
  // A gap that is rounding of the norm (equal eigenvalues) says nothing: the
  // quotient of two rounding errors would rotate by up to 1/8 at random and leave
  // the vectors orthonormal to 1e-10 only.
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * n;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / n), j = (int)(idx % n);
    double r = R[idx];
    const double num = S[idx] + lam[j] * r, dl = lam[j] - lam[i];
    double e;
    if (i != j && fabs(dl) > dmin && (fabs(dl) > delta || fabs(dl) > 8.0 * fabs(num))) e = num / dl;
    else e = 0.5 * r;
    E[idx] = e;
  }
}

__global__ void add_inplace_kernel(double* X, const double* Y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    X[i] += Y[i];
}

__global__ void i_minus_kernel(double* R, int n) {   // R <- I - R
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * n;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / n), j = (int)(idx % n);
    R[idx] = (i == j ? 1.0 : 0.0) - R[idx];
  }
}


static int elem_blocks(const LaCtx& la, long long n) {
  return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 8LL * la.sms));
}

// Ascending reorder of FP64 eigenpairs: Vout[:, rank(i)] = V[:, i], Wout[rank(i)] = lam[i].
// Ranks by integer comparison of order-preserving keys: n^2 FP64 comparisons hold the
// FP64 pipe (257 us at n = 580 with them, every block ranking all values).
__global__ void eig_sort64_kernel(const double* __restrict__ V, const double* __restrict__ lam, int n, double* Vout,
                                  double* Wout) {
  __shared__ unsigned long long key[kEighMax];
  __shared__ int rank[kEighMax];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(lam[i] + 0.0);   // -0 as +0
    key[i] = b >> 63 ? ~b : b | 1ull << 63;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const unsigned long long wi = key[i];
    int r = 0;
    for (int j = 0; j < n; ++j) r += key[j] < wi || (key[j] == wi && j < i);
    rank[i] = r;
  }
  __syncthreads();
  // every block ranks all n values, then moves its own rows
  for (int row = blockIdx.x; row < n; row += gridDim.x)
    for (int i = threadIdx.x; i < n; i += blockDim.x) Vout[(size_t)row * n + rank[i]] = V[(size_t)row * n + i];
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n; i += blockDim.x) Wout[rank[i]] = lam[i];
}

void eigh(const LaCtx& la, const double* A, int n, double* W, double* V, double* ws, int refine,
          const double* Vguess, bool skip_jacobi, int max_sweeps, int ns_steps) {
  if (n > kEighMax) throw RihfError(RIHF_ERR_INVALID_ARG, "eigensolver: order above its limit");
  int m = n + (n & 1);
  if (skip_jacobi && Vguess && refine > 0) {
    // Late SCF iterations: the previous eigenvectors are already close, so the
    // FP64 refinement alone converges (quadratically) without a Jacobi pass.
    double* d = ws + ((size_t)m * m + (size_t)n * m + m + 1) / 2;
    double* Vs = d + 4 * (size_t)n * n;   // the XE slot of the workspace
    double* lam = d + 6 * (size_t)n * n;
    RIHF_CUDA(cudaMemcpyAsync(V, Vguess, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, la.stream));
    eigh(la, A, n, W, V, ws, -refine, nullptr, false, max_sweeps, ns_steps);
    eig_sort64_kernel<<<std::min(n, 32), 256, 0, la.stream>>>(V, lam, n, Vs, W);
    RIHF_LAUNCH_CHECK();
    count(la);
    RIHF_CUDA(cudaMemcpyAsync(V, Vs, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, la.stream));
    return;
  }
  const bool refine_only = refine < 0;   // V already holds the starting vectors
  if (refine_only) refine = -refine;
  float* fA = reinterpret_cast<float*>(ws);
  float* fV = fA + (size_t)m * m;
  float* fW = fV + (size_t)n * m;
  double* d = ws + ((size_t)m * m + (size_t)n * m + m + 1) / 2;
  double* R = d;
  double* S = R + (size_t)n * n;
  double* AX = S + (size_t)n * n;
  double* E = AX + (size_t)n * n;
  double* XE = E + (size_t)n * n;
  double* Ag = XE + (size_t)n * n;
  double* lam = Ag + (size_t)n * n;
  double* sums = lam + n;
  const double* Ain = A;
  if (!refine_only && n > kJacobiMax) {
    tridiag_eigh(la, A, n, lam, XE, ws + eig_workspace_base(n));
    eig_sort64_kernel<<<std::min(n, 32), 256, 0, la.stream>>>(XE, lam, n, V, W);
    RIHF_LAUNCH_CHECK();
    count(la);
    refine = std::min(refine, kTridiagRefine);
  } else if (!refine_only) {
  if (Vguess) {
    // warm start: diagonalise Vg^T A Vg and rotate back
    GemmArgs g1;
    g1.M = n; g1.N = n; g1.K = n; g1.A = A; g1.lda = n; g1.B = Vguess; g1.ldb = n; g1.C = AX; g1.ldc = n;
    dgemm(la, g1);
    GemmArgs g2;
    g2.M = n; g2.N = n; g2.K = n; g2.A = Vguess; g2.lda = n; g2.transA = true; g2.B = AX; g2.ldb = n;
    g2.C = Ag; g2.ldc = n; g2.lower_only = g2.mirror = true;
    dgemm(la, g2);
    Ain = Ag;
  }
  // a looser stop (n eps) leaves close clusters too coarse for the FP64
  // refinement to separate
  jacobi(la, Ain, n, m, fA, fV, fW, max_sweeps, 2e-6f);
  eig_sort_kernel<<<std::min(n, 32), 256, 0, la.stream>>>(fV, fW, n, m, V, W);
  RIHF_LAUNCH_CHECK();
  count(la);
  if (Vguess) {
    // V <- Vguess * V
    GemmArgs g;
    g.M = n; g.N = n; g.K = n; g.A = Vguess; g.lda = n; g.B = V; g.ldb = n; g.C = XE; g.ldc = n;
    dgemm(la, g);
    RIHF_CUDA(cudaMemcpyAsync(V, XE, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, la.stream));
  }
  }   // Jacobi
  for (int it = 0; it < refine; ++it) {
    GemmArgs gr;   // R = V^T V
    gr.M = n; gr.N = n; gr.K = n; gr.A = V; gr.lda = n; gr.transA = true; gr.B = V; gr.ldb = n; gr.C = R; gr.ldc = n;
    gr.lower_only = gr.mirror = true;
    dgemm(la, gr);
    i_minus_kernel<<<elem_blocks(la, (long long)n * n), 256, 0, la.stream>>>(R, n);
    RIHF_LAUNCH_CHECK();
    GemmArgs ga;   // AX = A V
    ga.M = n; ga.N = n; ga.K = n; ga.A = A; ga.lda = n; ga.B = V; ga.ldb = n; ga.C = AX; ga.ldc = n;
    dgemm(la, ga);
    GemmArgs gs;   // S = V^T A V
    gs.M = n; gs.N = n; gs.K = n; gs.A = V; gs.lda = n; gs.transA = true; gs.B = AX; gs.ldb = n; gs.C = S; gs.ldc = n;
    gs.lower_only = gs.mirror = true;
    dgemm(la, gs);
    oa_lambda_kernel<<<elem_blocks(la, n), 256, 0, la.stream>>>(R, S, n, lam);
    // partial norms in the XE slot (written only by the update GEMM below)
    const int nparts = (int)std::max<long long>(1, std::min<long long>(kOaParts, (long long)n * n / 1024));
    double* part = (long long)n * n >= 3LL * nparts ? XE : sums;   // sums: 8 doubles, enough for one part
    oa_norms_kernel<<<nparts, 256, 0, la.stream>>>(R, S, A, lam, n, part);
    oa_e_kernel<<<elem_blocks(la, (long long)n * n), 256, 0, la.stream>>>(R, S, lam, part, nparts, n, E);
    RIHF_LAUNCH_CHECK();
    GemmArgs ge;   // XE = V E ; V += XE
    ge.M = n; ge.N = n; ge.K = n; ge.A = V; ge.lda = n; ge.B = E; ge.ldb = n; ge.C = XE; ge.ldc = n;
    dgemm(la, ge);
    add_inplace_kernel<<<elem_blocks(la, (long long)n * n), 256, 0, la.stream>>>(V, XE, (long long)n * n);
    RIHF_LAUNCH_CHECK();
    count(la, 5);
  }
  if (refine > 0) {
    RIHF_CUDA(cudaMemcpyAsync(W, lam, sizeof(double) * n, cudaMemcpyDeviceToDevice, la.stream));
    // Newton-Schulz re-orthonormalisation V <- V (3I - V^T V)/2: columns inside
    // near-degenerate clusters are only orthonormalised to first order by the
    // refinement's r_ij/2 rule; two quadratic steps take V^T V to I.
    for (int it = 0; it < ns_steps; ++it) {
      GemmArgs gr;
      gr.M = n; gr.N = n; gr.K = n; gr.A = V; gr.lda = n; gr.transA = true; gr.B = V; gr.ldb = n; gr.C = R;
      gr.ldc = n; gr.alpha = -0.5; gr.lower_only = gr.mirror = true;
      dgemm(la, gr);
      identity(la, E, n);
      axpby(la, n * n, 1.0, R, 1.5, E, R);
      GemmArgs gv;
      gv.M = n; gv.N = n; gv.K = n; gv.A = V; gv.lda = n; gv.B = R; gv.ldb = n; gv.C = XE; gv.ldc = n;
      dgemm(la, gv);
      RIHF_CUDA(cudaMemcpyAsync(V, XE, sizeof(double) * n * n, cudaMemcpyDeviceToDevice, la.stream));
    }
  }
}

// ------------------------------------------------------------ elementwise

__global__ void axpby_kernel(long long n, double a, const double* x, double b, const double* y, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = a * x[i] + b * y[i];
}
void axpby(const LaCtx& la, int n, double a, const double* x, double b, const double* y, double* out) {
  axpby_kernel<<<elem_blocks(la, n), 256, 0, la.stream>>>(n, a, x, b, y, out);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void add3_kernel(long long n, const double* x, const double* y, const double* z, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = x[i] + y[i] + z[i];
}
void add3(const LaCtx& la, int n, const double* x, const double* y, const double* z, double* out) {
  add3_kernel<<<elem_blocks(la, n), 256, 0, la.stream>>>(n, x, y, z, out);
  RIHF_LAUNCH_CHECK();
  count(la);
}

// Deterministic single-block reductions (n up to a few million).
__global__ void dot_kernel(long long n, const double* x, const double* y, double* out) {
  __shared__ double r[32];
  double s = 0.0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) s += x[i] * y[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) r[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) t += r[w];
    *out = t;
  }
}
void dot(const LaCtx& la, int n, const double* x, const double* y, double* out) {
  dot_kernel<<<1, 1024, 0, la.stream>>>(n, x, y, out);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void scale_copy_kernel(long long n, double a, const double* x, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = a * x[i];
}
void scale_copy(const LaCtx& la, int n, double a, const double* x, double* out) {
  scale_copy_kernel<<<elem_blocks(la, n), 256, 0, la.stream>>>(n, a, x, out);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void antisym_kernel(const double* A, double* C, int n) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)n * n;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / n), j = (int)(idx % n);
    C[idx] = A[idx] - A[(size_t)j * n + i];
  }
}
void antisym(const LaCtx& la, const double* A, double* C, int n) {
  antisym_kernel<<<elem_blocks(la, (long long)n * n), 256, 0, la.stream>>>(A, C, n);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void copy_cols_kernel(const double* src, int nrows, int ld, int ncol, double s, double* dst) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)nrows * ncol;
       idx += (long long)gridDim.x * blockDim.x) {
    int i = (int)(idx / ncol), j = (int)(idx % ncol);
    dst[idx] = s * src[(size_t)i * ld + j];
  }
}
void copy_cols(const LaCtx& la, const double* src, int nrows, int ld, int ncol, double s, double* dst) {
  copy_cols_kernel<<<elem_blocks(la, (long long)nrows * ncol), 256, 0, la.stream>>>(src, nrows, ld, ncol, s, dst);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void transpose_kernel(const double* __restrict__ src, int rows, int cols, double* __restrict__ dst) {
  __shared__ double t[32][33];
  int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int i = r0 + r, j = c0 + threadIdx.x;
    t[r][threadIdx.x] = (i < rows && j < cols) ? src[(size_t)i * cols + j] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int i = c0 + r, j = r0 + threadIdx.x;   // dst row i (source column), dst column j (source row)
    if (i < cols && j < rows) dst[(size_t)i * rows + j] = t[threadIdx.x][r];
  }
}
void transpose(const LaCtx& la, const double* src, int rows, int cols, double* dst) {
  transpose_kernel<<<dim3(ceil_div(cols, 32), ceil_div(rows, 32)), dim3(32, 8), 0, la.stream>>>(src, rows, cols, dst);
  RIHF_LAUNCH_CHECK();
  count(la);
}

__global__ void scale_cols_kernel(const double* X, const double* v, int nrows, int ncol, double* out) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < (long long)nrows * ncol;
       idx += (long long)gridDim.x * blockDim.x)
    out[idx] = X[idx] * v[idx % ncol];
}
void scale_cols(const LaCtx& la, const double* X, const double* v, int nrows, int ncol, double* out) {
  scale_cols_kernel<<<elem_blocks(la, (long long)nrows * ncol), 256, 0, la.stream>>>(X, v, nrows, ncol, out);
  RIHF_LAUNCH_CHECK();
  count(la);
}

}  // namespace rihf
