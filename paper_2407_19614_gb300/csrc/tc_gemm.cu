// BF16 digit-plane GEMM on the 5th-generation tensor cores (tcgen05 + TMEM),
// operands staged in shared memory by bulk asynchronous copies.  See
// tc_gemm.cuh for the number format.
#include <algorithm>
#include <cmath>

#include "../../include/rihf.h"
#include "tc_gemm.cuh"

namespace rihf {

namespace {

constexpr int kOzThreads = 256;                                  // slicing kernel
constexpr int kPlaneElems = kOzTileM * kOzChunk;                // 4096 BF16 = 8 KB
constexpr int kMaxChunksPerBlock = kOzMaxChunksPerBlock;
constexpr int kCoreK = kOzChunk / 8;                             // core matrices along K per chunk
constexpr unsigned long long kWaitNs = 2000000000ULL;     // bounded waits: 2 s

// ------------------------------------------------------------ PTX wrappers

__device__ inline uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ inline void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Spin on an mbarrier phase with a wall-clock limit; false when it ran out.
__device__ inline bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > kWaitNs) return false;
  }
}

__device__ inline void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ inline void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D (TMEM) = A (smem) . B (smem)^T [+ D], BF16 inputs, FP32 accumulator; issued by
// the one lane of the warp with lead != 0 (a predicate, so that the warp stays
// converged and the operands stay in uniform registers).
__device__ inline void mma_bf16(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc,
                                uint32_t lead) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(lead)
      : "memory");
}

__device__ inline void mma_commit(uint64_t* bar, uint32_t lead) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_addr(bar)),
      "r"(lead)
      : "memory");
}

// 32 lanes x 4 consecutive 32-bit columns; thread i gets lane (base + i).
__device__ inline void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}

__device__ inline void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One 32-byte sector of a row (p 32-byte aligned).
__device__ inline void st_sector(double* p, const double* v) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "d"(v[0]), "d"(v[1]),
               "d"(v[2]), "d"(v[3])
               : "memory");
}

// Shared-memory matrix descriptor, no swizzle, K-major core matrices of
// 8 rows x 16 bytes: 128 B between K-adjacent core matrices (leading byte
// offset), kCoreK * 128 B between 8-row groups (stride byte offset), version 1.
__device__ inline uint64_t smem_desc(uint32_t addr) {
  const uint64_t base = ((uint64_t)(128 >> 4) << 16) | ((uint64_t)((kCoreK * 128) >> 4) << 32) | (1ULL << 46);
  return base | (uint64_t)((addr & 0x3FFFF) >> 4);
}

// ------------------------------------------------------------ number format

// x as a signed fixed-point integer V = x * 2^{1077 - E} (|V| < 2^55 when E is
// the largest biased exponent of the block), rounded to nearest.
__device__ inline long long oz_fixed(double x, int E) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7FF);
  if (e == 0 || E == 0) return 0;
  const long long mant = (long long)((bits & ((1ULL << 52) - 1)) | (1ULL << 52));
  const int sh = E - e - 2;
  long long V;
  if (sh < 0) V = mant << (-sh);
  else if (sh == 0) V = mant;
  else if (sh < 62) V = (mant + (1LL << (sh - 1))) >> sh;
  else V = 0;
  return (bits >> 63) ? -V : V;
}

// S * 2^e2 as the nearest double (ties to even), 0 below the normal range: integer
// construction, no FP64 arithmetic and no branches, so that the conversions of
// a thread's elements overlap.
__device__ inline double oz_to_double(long long S, int e2) {
  const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int lz = __clzll((long long)a);                     // 64 when S = 0
  const unsigned long long n = a << (lz & 63);
  // mantissa with its leading bit (53 bits), rounded; a carry out of it moves
  // into the exponent field by the addition below
  const unsigned long long m = (n >> 11) + ((n & 0x7FF) + ((n >> 11) & 1) > 0x400 ? 1ULL : 0ULL);
  const int be = 63 - lz + e2 + 1023;                        // biased exponent before a carry
  unsigned long long bits = ((unsigned long long)(uint32_t)(be - 1) << 52) + m;
  const int bc = be + (int)(m >> 53);
  if (bc <= 0 || S == 0) bits = 0ULL;
  if (bc >= 2047 && S != 0) bits = 0x7FFULL << 52;
  if (S < 0 && bc > 0) bits |= 1ULL << 63;
  return __longlong_as_double((long long)bits);
}

// ------------------------------------------------------------ slicing

// Element (r, k) of the operand is X[r*s_r + (k % KR)*s_k1 + (k / KR)*s_k2].
struct OzSrc {
  const double* X;
  int rows, K;
  long long s_r, s_k1, s_k2;
  int KR;
  int RR;             // > 0: rows split as (r % RR, r / RR) with strides s_r, s_r2
  long long s_r2;
  int PN;             // > 0: pair-packed symmetric PN x PN matrices, s_r2 apart:
                      // row r = (matrix r / PN, mu = r % PN), column k = nu
  int vec;            // 8-element runs are contiguous, 16-byte aligned and whole or empty
};

// The elements k0 .. k0+7 of row r (zero outside the operand).
__device__ inline void oz_load8(const OzSrc& S, int r, int k0, double (&x)[8]) {
  if (r >= S.rows || k0 >= S.K) {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = 0.0;
  } else if (S.PN > 0) {
    const double* p = S.X + (long long)(r / S.PN) * S.s_r2;
    const int mu = r % S.PN;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = k0 + e, a = max(mu, k), b = min(mu, k);
      x[e] = k < S.K ? p[(long long)a * (a + 1) / 2 + b] : 0.0;
    }
  } else {
    int q = 0, m = k0;
    if (S.KR < S.K) {
      q = k0 / S.KR;
      m = k0 - q * S.KR;
    }
    const double* p = S.X + (S.RR > 0 ? (long long)(r % S.RR) * S.s_r + (long long)(r / S.RR) * S.s_r2
                                      : (long long)r * S.s_r);
    if (S.vec) {
      const double2* v = reinterpret_cast<const double2*>(p + (long long)q * S.s_k2 + m);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double2 t = v[e];
        x[2 * e] = t.x;
        x[2 * e + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        x[e] = k0 + e < S.K ? p[(long long)q * S.s_k2 + (long long)m * S.s_k1] : 0.0;
        if (++m == S.KR) {
          m = 0;
          ++q;
        }
      }
    }
  }
}

__device__ inline int oz_emax8(const double (&x)[8]) {
  int e = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) e = max(e, (__double2hiint(x[i]) >> 20) & 0x7FF);
  return e;
}

// The digits of eight elements, 16 bytes per plane (planes kPlaneElems apart).  With
// q_t = V / 2^(48 - 8t) rounded half up, digit t is q_t - 256 q_{t-1}, in 32-bit
// arithmetic modulo 2^32; 0x4B400000 + d is the FP32 number 1.5 2^23 + d, and the
// upper half of the difference to 1.5 2^23 is the BF16.
__device__ inline void oz_digits8(const double (&x)[8], int emax, int smax, uint16_t* dst) {
  uint32_t lo[8], hi[8], prev[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned long long V = (unsigned long long)oz_fixed(x[e], emax);
    lo[e] = (uint32_t)V;
    hi[e] = (uint32_t)(V >> 32);
    prev[e] = 0u;
  }
#pragma unroll
  for (int t = 0; t < kOzMaxDigits; ++t) {
    if (t >= smax) break;
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      uint32_t q;
      if (t == 0) q = (uint32_t)((int)(hi[e] + 0x8000u) >> 16);
      else if (t == 1) q = (uint32_t)((int)(hi[e] + 0x80u) >> 8);
      else if (t == 2) q = hi[e] + (lo[e] >> 31);
      else if (t < 6) q = __funnelshift_r(lo[e], hi[e], 48 - 8 * t) + ((lo[e] >> (47 - 8 * t)) & 1u);
      else q = lo[e];
      const uint32_t d = q - 256u * prev[e];
      prev[e] = q;
      w[e] = __float_as_uint(__uint_as_float(0x4B400000u + d) - 12582912.0f);
    }
    *reinterpret_cast<uint4*>(dst + (size_t)t * kPlaneElems) =
        make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632), __byte_perm(w[4], w[5], 0x7632),
                   __byte_perm(w[6], w[7], 0x7632));
  }
}

// Exponents and digit planes of one K block (blockIdx.y) in one launch: a warp holds
// eight rows of one chunk (lane = row, 8-element run j: its stores of a digit are
// 512 contiguous bytes), `slots` warps of the block share the same rows and step
// through the block's chunks, and exchange their exponents through shared memory.
// The first kHeld chunks of a warp stay in registers, the others are read again
// (from L1 or L2).  exps[r * nkb + kb] = largest biased exponent of row r over
// K block kb.  Bound by the store of the planes (14 bytes an element at 7 digits).
// Two passes over memory before: exponents by atomicMax into a zeroed array, then
// the digits, 76 + 194 us for 162816 x 192.
constexpr int kHeld = 2;

__global__ void __launch_bounds__(kOzThreads) oz_slice_kernel(OzSrc S, int kchunks, int smax, int kb_chunks, int nkb,
                                                              int slots, int* __restrict__ exps,
                                                              uint16_t* __restrict__ planes) {
  constexpr int kWarps = kOzThreads / 32;
  __shared__ int se[kWarps][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = warp % slots, rg = warp / slots;
  const int r = (blockIdx.x * (kWarps / slots) + rg) * 8 + (lane >> 2);
  const int j = lane & 3;
  const int kb = blockIdx.y, c0 = kb * kb_chunks + slot, c1 = min((kb + 1) * kb_chunks, kchunks);
  double x[kHeld][8];
  int emax = 0;
#pragma unroll
  for (int h = 0; h < kHeld; ++h) {
    const int c = c0 + h * slots;
    if (c < c1) {
      oz_load8(S, r, c * kOzChunk + 8 * j, x[h]);
      emax = max(emax, oz_emax8(x[h]));
    }
  }
  for (int c = c0 + kHeld * slots; c < c1; c += slots) {
    double y[8];
    oz_load8(S, r, c * kOzChunk + 8 * j, y);
    emax = max(emax, oz_emax8(y));
  }
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 1));
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 2));
  if (j == 0) se[warp][lane >> 2] = emax;
  __syncthreads();
  for (int k = 0; k < slots; ++k) emax = max(emax, se[rg * slots + k][lane >> 2]);
  if (slot == 0 && j == 0) exps[(size_t)r * nkb + kb] = emax;
  const int rt = r / kOzTileM, rr = r % kOzTileM;
  uint16_t* dst = planes + (size_t)rt * kchunks * smax * kPlaneElems + (rr / 8) * (kCoreK * 64) + j * 64 + (rr % 8) * 8;
#pragma unroll
  for (int h = 0; h < kHeld; ++h) {
    const int c = c0 + h * slots;
    if (c < c1) oz_digits8(x[h], emax, smax, dst + (size_t)c * smax * kPlaneElems);
  }
  for (int c = c0 + kHeld * slots; c < c1; c += slots) {
    double y[8];
    oz_load8(S, r, c * kOzChunk + 8 * j, y);
    oz_digits8(y, emax, smax, dst + (size_t)c * smax * kPlaneElems);
  }
}

// ------------------------------------------------------------ GEMM
//
// Persistent, warp-specialised kernel (one CTA per SM: it holds all 512 TMEM
// columns).  Work items are (row tile, column tile, K block) triples taken from
// a global counter, so tiles that the symmetry options skip cost nothing and
// the SMs stay balanced.
//   warp 17 (one lane): takes items, streams their K chunks' digit planes into
//     a ring of shared-memory stages with bulk copies;
//   warp 16: issues the MMAs of each chunk and commits stage releases and, every
//     G chunks, a full accumulator group;
//   warps 0-15: drain the s TMEM accumulators of each group (a row and a quarter
//     of the columns per thread) into int64 fixed-point sums; the group is released when
//     its last columns are in registers, so the next group's MMAs overlap the
//     rest of the conversion and, at a tile's end, the stores.
// The kernel is compiled per digit count and column tile: every descriptor offset
// and diagonal weight is then a constant.  With run-time counts one MMA took 138
// clocks to issue (its table entry, its operands' way into uniform registers)
// against the 90 it runs, a tile's diagonals 4.8 k clocks to read (now 2.4 k) and
// its epilogue 20 k (now 12 k: no FP64 product for alpha = +-2^n, exponents
// fetched ahead, 32-byte stores); 77824 x 64, K = 384, 7 digits: 303 -> 212 k
// clocks a CTA, the tensor pipe active 30 -> 41 %.  What remains is the read-out
// between groups, which the 512 TMEM columns leave no room to overlap, and for
// operands from HBM the two stages that shared memory holds.
// A group spans G = floor(1024 / s) / kOzChunk chunks: every diagonal sum then
// stays below s * 32G * 128^2 <= 2^24 and is exact in FP32.  Every wait is
// bounded; the first one that runs out raises a shared abort flag, all roles
// leave, the copies and MMAs still in flight are awaited (bounded) and
// la.flag[1] is set.

// Four drain warps a scheduler: the read-out and the epilogue are chains of integer
// instructions that two warps did not cover (a gradient's Y at 580 orbitals, whose
// tiles are two chunks long and all epilogue, 8.9 -> 8.3 ms; K at 384 orbitals 3 to 5 %).
constexpr int kDrainThreads = 512;
constexpr int kMmaWarp = kDrainThreads / 32, kCopyWarp = kMmaWarp + 1;
constexpr int kGemmThreads = kDrainThreads + 64;
constexpr int kMaxStages = 4;
constexpr int kItemSlots = 2;
constexpr int kTmemCols = 512;
constexpr int kSmemMax = 227 * 1024;
constexpr int kSmemMin = 116 * 1024;   // more than half an SM's shared memory: one CTA per SM
constexpr int kBookBytes = 1024;

struct OzBook {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t accfull, accempty;
  uint64_t item_full[kItemSlots], item_empty[kItemSlots];
  int item[kItemSlots];
  uint32_t tslot;
  int abort;
  int issued, consumed;
  int dwait[2];        // the drain poller's wait results, alternating slots
};
static_assert(sizeof(OzBook) <= kBookBytes, "bookkeeping block");

struct OzTiling {
  int M, N, TN, mtiles, ntiles, nsplit, nitems, nfast;
  int lower_only, symcols, kb_chunks, kchunks;
  int s, G, nst, stage_bytes;
  int aexp, aneg, scale;   // alpha = +-2^aexp (scale 0), or it is multiplied
};

__device__ inline void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Wait for a phase; false if the shared abort flag is up or the time ran out
// (which raises the flag).
__device__ inline bool oz_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    if (global_ns() - t0 > kWaitNs) {
      *abort = 1;
      return false;
    }
  }
}

__device__ inline void oz_decode(const OzTiling& T, int idx, int& mt, int& nt, int& split, int& c0, int& c1) {
  split = idx % T.nsplit;
  const int tile = idx / T.nsplit;
  if (T.nfast) {
    nt = tile % T.ntiles;
    mt = tile / T.ntiles;
  } else {
    mt = tile % T.mtiles;
    nt = tile / T.mtiles;
  }
  c0 = split * T.kb_chunks;
  c1 = min(c0 + T.kb_chunks, T.kchunks);
}

// Whether an item has work: a non-empty K range, a tile that meets the lower
// triangle (lower_only), a column tile with a needed column (symcols).
__device__ inline bool oz_valid(const OzTiling& T, int mt, int nt, int c0, int c1) {
  if (c0 >= c1) return false;
  if (T.lower_only && mt * kOzTileM + kOzTileM - 1 < nt * T.TN) return false;
  if (T.symcols > 0) {
    // columns n = a * symcols + b are needed when b <= a; a range inside one
    // a holds b from n0 % symcols up, a range across two holds b = 0
    const int n0 = nt * T.TN, n1 = min(n0 + T.TN, T.N) - 1;
    const int a0 = n0 / T.symcols;
    if (n1 / T.symcols == a0 && n0 % T.symcols > a0) return false;
  }
  return true;
}

// Columns that a drain warp passes through shared memory at a time when it adds to C.
template <int TN>
constexpr int kStageCols = TN % 32 == 0 ? 8 : 4;

// The integer in accumulator d (d + 1 digit pairs of at most 2^14 K'(S) each): by an
// FP32 addition where that stays within 2^22, else by a conversion instruction,
// which only the slow unit has (16 a clock and SM: the read-out is bound by it).
template <int S>
__device__ inline int oz_sum_to_int(int d, float x) {
  constexpr int kp = (1024 / S) / kOzChunk * kOzChunk;   // elements accumulated between read-outs
  if ((d + 1) * kp <= 256) return __float_as_int(x + 12582912.0f) - 0x4B400000;
  return __float2int_rn(x);
}

template <int S, int TN>
__global__ void __launch_bounds__(kGemmThreads, 1)
    oz_gemm_kernel(OzOperand A, OzOperand B, OzTiling T, double alpha, double* C, long long MR, long long cs_m1,
                   long long cs_m2, long long cs_n, int atomic, int* flag, int* sched) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  OzBook* bk = reinterpret_cast<OzBook*>(smem + (size_t)T.nst * T.stage_bytes);
  volatile int* abort = &bk->abort;
  // the warp index by a shuffle: the roles' branches are then known to be uniform
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  constexpr uint32_t s = S, a_bytes = s * kPlaneElems * 2, b_plane = TN * kOzChunk * 2;

  if (tid == 0) {
    for (int i = 0; i < T.nst; ++i) {
      mbar_init(&bk->full[i], 1);
      mbar_init(&bk->empty[i], 1);
    }
    mbar_init(&bk->accfull, 1);
    // one arrival per drain warp (its lane 0, after the warp's reads)
    mbar_init(&bk->accempty, kDrainThreads / 32);
    for (int k = 0; k < kItemSlots; ++k) {
      mbar_init(&bk->item_full[k], 1);
      mbar_init(&bk->item_empty[k], kDrainThreads / 32 + 1);
    }
    bk->abort = 0;
    bk->issued = bk->consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc(&bk->tslot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = bk->tslot;

  if (warp == kCopyWarp) {
    if (lane == 0) {   // ---------------- producer
      uint32_t i = 0;
      bool ok = true;
      for (int q = 0; ok; ++q) {
        int idx, mt = 0, nt = 0, split = 0, c0 = 0, c1 = 0;
        for (;;) {
          idx = atomicAdd(sched, 1);
          if (idx >= T.nitems) break;
          oz_decode(T, idx, mt, nt, split, c0, c1);
          if (oz_valid(T, mt, nt, c0, c1)) break;
        }
        const int slot = q % kItemSlots;
        if (q >= kItemSlots && !oz_wait(&bk->item_empty[slot], ((q / kItemSlots) - 1) & 1, abort)) break;
        bk->item[slot] = idx < T.nitems ? idx : -1;
        mbar_arrive(&bk->item_full[slot]);
        if (idx >= T.nitems) break;
        const int b_rt = (nt * TN) / kOzTileM, b_off = (nt * TN) % kOzTileM;
        for (int c = c0; c < c1; ++c, ++i) {
          const int st = (int)(i % (uint32_t)T.nst);
          if (i >= (uint32_t)T.nst && !oz_wait(&bk->empty[st], ((i / T.nst) - 1) & 1, abort)) {
            ok = false;
            break;
          }
          uint8_t* As = smem + (size_t)st * T.stage_bytes;
          uint8_t* Bs = As + a_bytes;
          mbar_expect_tx(&bk->full[st], a_bytes + (uint32_t)s * b_plane);
          bulk_load(As, A.planes + ((size_t)mt * A.kchunks + c) * A.smax * kPlaneElems, a_bytes, &bk->full[st]);
          for (uint32_t u = 0; u < s; ++u)
            bulk_load(Bs + u * b_plane,
                      B.planes + (((size_t)b_rt * B.kchunks + c) * B.smax + u) * kPlaneElems +
                          (size_t)b_off * kOzChunk,
                      b_plane, &bk->full[st]);
        }
      }
      bk->issued = (int)i;
      // every CTA counts itself once it takes no more items; the last one
      // resets the counters for the next launch on this stream
      __threadfence();
      if (atomicAdd(sched + 1, 1) == (int)gridDim.x - 1) {
        atomicExch(sched, 0);
        atomicExch(sched + 1, 0);
      }
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ---------------- MMA issuer: the warp stays converged, lane 0 issues
    // BF16 x BF16 -> FP32, M = 128; N is set per MMA
    const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kOzTileM >> 4) << 24);
    constexpr int planes_per_mma = 256 / TN;
    const uint32_t lead = lane == 0 ? 1u : 0u;
    // a wait whose result the lanes agree on
    auto wait_all = [&](uint64_t* bar, uint32_t parity) -> bool {
      return __all_sync(0xffffffffu, oz_wait(bar, parity, abort));
    };
    uint32_t i = 0, grp = 0;
    int last_st = -1;
    uint32_t last_par = 0;
    bool ok = true;
    for (int q = 0; ok; ++q) {
      const int slot = q % kItemSlots;
      if (!wait_all(&bk->item_full[slot], (q / kItemSlots) & 1)) break;
      const int idx = __shfl_sync(0xffffffffu, *(volatile int*)&bk->item[slot], 0);
      if (lane == 0) mbar_arrive(&bk->item_empty[slot]);
      if (idx < 0) break;
      int mt, nt, split, c0, c1;
      oz_decode(T, idx, mt, nt, split, c0, c1);
      for (int c = c0; c < c1; ++c, ++i) {
        const int st = (int)(i % (uint32_t)T.nst);
        if (!wait_all(&bk->full[st], (i / T.nst) & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const bool first = (c - c0) % T.G == 0, last = (c - c0) % T.G == T.G - 1 || c == c1 - 1;
        if (first && grp > 0) {   // the last group read out
          if (!wait_all(&bk->accempty, (grp - 1) & 1)) {
            ok = false;
            ++i;
            break;
          }
          tc_fence_after();
        }
        // per K step j, A plane t and group of B planes, one MMA; the B planes
        // u = 1..s+1-t lie one after another in shared memory with the same
        // 8-row-group stride, so up to 256 / TN of them form one operand of
        // N = count * TN rows, and the product (t, u) lands on the columns of
        // anti-diagonal t + u.  Plane and K-step offsets go into the 14-bit
        // address field of the stage's descriptors (shared addresses stay
        // below 256 KB).
        const uint32_t a_s = smem_addr(smem + (size_t)st * T.stage_bytes);
        const uint64_t a_d0 = smem_desc(a_s), b_d0 = smem_desc(a_s + a_bytes);
#pragma unroll
        for (int j = 0; j < kOzChunk / 16; ++j) {
#pragma unroll
          for (int t = 0; t < S; ++t) {
            const uint64_t a_d = a_d0 + (uint64_t)((t * kPlaneElems * 2 + j * 256) >> 4);
            const uint32_t acc = t == 0 && j == 0 && first ? 0u : 1u;
#pragma unroll
            for (int u = 0; u < S - t; u += planes_per_mma) {
              constexpr int most = planes_per_mma;
              const int np = most < S - t - u ? most : S - t - u;
              mma_bf16(taddr + (uint32_t)((t + u) * TN), a_d, b_d0 + (uint64_t)((u * (int)b_plane + j * 256) >> 4),
                       idesc0 | ((uint32_t)((np * TN) >> 3) << 17), acc, lead);
            }
          }
        }
        mma_commit(&bk->empty[st], lead);   // the stage is free once these MMAs are done
        last_st = st;
        last_par = (i / T.nst) & 1;
        if (last) {
          mma_commit(&bk->accfull, lead);
          ++grp;
        }
      }
    }
    if (lane == 0) bk->consumed = (int)i;
    if (*abort && last_st >= 0) mbar_wait(&bk->empty[last_st], last_par);   // MMAs in flight
    __syncwarp();
  } else {   // ---------------- drain: warps 0-15
    const int row = 32 * (warp & 3) + lane;
    constexpr int ncol = TN / 4;   // a row and a quarter of the columns per thread
    const int col0 = (warp >> 2) * ncol;
    const uint32_t t_row = taddr + ((uint32_t)(32 * (warp & 3)) << 16);
    // one thread polls, the other drain threads wait on a hardware named
    // barrier (spinning 512 threads would compete with the copy and MMA
    // threads for issue slots and for the barrier unit); the poller is lane 0
    // of warp 2, on a scheduler that neither the MMA nor the copy warp uses
    int nwait = 0;
    auto drain_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      const int k = nwait++ & 1;
      if (tid == 64) bk->dwait[k] = oz_wait(bar, parity, abort) ? 1 : 0;
      asm volatile("bar.sync 1, %0;" ::"r"(kDrainThreads) : "memory");
      return *(volatile int*)&bk->dwait[k] != 0;
    };
    uint32_t grp = 0;
    for (int q = 0;; ++q) {
      const int slot = q % kItemSlots;
      bool ok = drain_wait(&bk->item_full[slot], (q / kItemSlots) & 1);
      if (!ok) break;
      const int idx = *(volatile int*)&bk->item[slot];
      __syncwarp();
      if (lane == 0) mbar_arrive(&bk->item_empty[slot]);
      if (idx < 0) break;
      int mt, nt, split, c0, c1;
      oz_decode(T, idx, mt, nt, split, c0, c1);
      // the exponents (padded to whole tiles) are fetched ahead of their use:
      // lane k's eb is that of column k of the warp's ncol <= 16
      const int m = mt * kOzTileM + row, n0 = nt * TN + col0;
      const int ea = A.exps[(size_t)m * A.nkb + split] - 2095 + T.aexp;
      const int eb = lane < ncol ? B.exps[(size_t)(n0 + lane) * B.nkb + split] : 0;
      long long acc[ncol];
#pragma unroll
      for (int k = 0; k < ncol; ++k) acc[k] = 0;
      for (int c = c0; c < c1 && ok; c += T.G) {
        ok = drain_wait(&bk->accfull, grp & 1);
        if (!ok) break;
        tc_fence_after();
        // four columns of all s diagonals at a time (the warp's last block read
        // frees the accumulators): the element's sum then has constant weights
        // 2^37, 2^29, ... 2^-11, one multiply-add each
#pragma unroll
        for (int q4 = 0; q4 < ncol / 4; ++q4) {
          uint32_t r[S][4];
#pragma unroll
          for (int d = 0; d < S; ++d) tmem_ld4(t_row + (uint32_t)(d * TN + col0 + 4 * q4), r[d]);
          tmem_wait_ld();
          if (q4 == ncol / 4 - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bk->accempty);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            long long a = acc[4 * q4 + e];
            int low = 0;
#pragma unroll
            for (int d = 0; d < S; ++d) {
              const int v = oz_sum_to_int<S>(d, __uint_as_float(r[d][e]));
              const int sh = 37 - 8 * d;
              if (sh >= 0) a += (long long)v * (1LL << (sh < 0 ? 0 : sh));
              else low += v >> (sh < 0 ? -sh : 0);
            }
            if (S > 5) a += low;
            acc[4 * q4 + e] = a;
          }
        }
        ++grp;
      }
      if (!ok) break;
      // all of the thread's values first, then the stores
      const int nv = min(ncol, T.N - n0);
      double v[ncol];
#pragma unroll
      for (int k = 0; k < ncol; ++k)
        v[k] = oz_to_double(T.aneg ? -acc[k] : acc[k], ea + __shfl_sync(0xffffffffu, eb, k));
      if (T.scale)   // not a predicate on each product: those hold the FP64 pipe also when it is false
#pragma unroll
        for (int k = 0; k < ncol; ++k) v[k] *= alpha;
      const int mr = MR < T.M ? (int)MR : T.M;
      double* dst = C + (long long)(m % mr) * cs_m1 + (long long)(m / mr) * cs_m2 + (long long)n0 * cs_n;
      // whole 32-byte sectors when the row is contiguous and aligned (16-byte halves
      // write a sector twice)
      const bool sectors =
          __all_sync(0xffffffffu, m >= T.M || (cs_n == 1 && nv == ncol && ((uintptr_t)dst & 31) == 0));
      if (atomic == 2 && cs_n == 1) {
        // added to: the warp's 32 rows go through shared memory, W columns at a time,
        // so that 32 / W whole row segments are read and written at once
        constexpr int W = kStageCols<TN>, RP = 32 / W;
        double* stg = reinterpret_cast<double*>(smem + (size_t)T.nst * T.stage_bytes + kBookBytes) + warp * 32 * (W + 1);
        const int cc = lane % W, rr = lane / W, m0 = mt * kOzTileM + 32 * (warp & 3);
#pragma unroll
        for (int k0 = 0; k0 < ncol; k0 += W) {
          __syncwarp();
#pragma unroll
          for (int k = 0; k < W; ++k) stg[lane * (W + 1) + k] = v[k0 + k];
          __syncwarp();
          double old[W];
#pragma unroll
          for (int i = 0; i < W; ++i) {
            const int q = i * RP + rr;
            const double* p =
                reinterpret_cast<const double*>(__shfl_sync(0xffffffffu, (unsigned long long)(uintptr_t)dst, q));
            old[i] = m0 + q < T.M && k0 + cc < nv ? p[k0 + cc] : 0.0;
          }
#pragma unroll
          for (int i = 0; i < W; ++i) {
            const int q = i * RP + rr;
            double* p = reinterpret_cast<double*>(__shfl_sync(0xffffffffu, (unsigned long long)(uintptr_t)dst, q));
            const double sum = old[i] + stg[q * (W + 1) + cc];
            if (m0 + q < T.M && k0 + cc < nv) p[k0 + cc] = sum;
          }
        }
      } else if (m < T.M) {
        if (atomic == 1) {
#pragma unroll
          for (int k = 0; k < ncol; ++k)
            if (k < nv) atomicAdd(dst + (long long)k * cs_n, v[k]);
        } else if (sectors && atomic == 0) {
#pragma unroll
          for (int k0 = 0; k0 < ncol; k0 += 4) st_sector(dst + k0, v + k0);
        } else if (cs_n == 1 && ((uintptr_t)dst & 15) == 0) {
          double2* d2 = reinterpret_cast<double2*>(dst);
#pragma unroll
          for (int k = 0; k < ncol / 2; ++k) {
            if (2 * k + 1 < nv) d2[k] = make_double2(v[2 * k], v[2 * k + 1]);
            else if (2 * k < nv) dst[2 * k] = v[2 * k];
          }
        } else {
#pragma unroll
          for (int k = 0; k < ncol; ++k) {
            if (k < nv) {
              double* d = dst + (long long)k * cs_n;
              if (atomic == 2) *d += v[k];
              else *d = v[k];
            }
          }
        }
      }
    }
  }

  __syncthreads();
  if (*abort) {
    if (warp == kCopyWarp && lane == 0) {
      // copies still in flight: chunks issued but never consumed
      for (int i = bk->consumed; i < bk->issued; ++i) mbar_wait(&bk->full[i % T.nst], (i / T.nst) & 1);
    }
    if (tid == 0) atomicOr(flag + 1, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(taddr, kTmemCols);
  }
}

using OzKernel = void (*)(OzOperand, OzOperand, OzTiling, double, double*, long long, long long, long long, long long,
                          int, int*, int*);

template <int S>
OzKernel oz_kernel_tn(int tn) {
  return tn <= 16 ? oz_gemm_kernel<S, 16> : tn <= 32 ? oz_gemm_kernel<S, 32> : tn <= 48 ? oz_gemm_kernel<S, 48>
                                                                                   : oz_gemm_kernel<S, 64>;
}

OzKernel oz_kernel(int s, int tn) {
  switch (s) {
    case 1: return oz_kernel_tn<1>(tn);
    case 2: return oz_kernel_tn<2>(tn);
    case 3: return oz_kernel_tn<3>(tn);
    case 4: return oz_kernel_tn<4>(tn);
    case 5: return oz_kernel_tn<5>(tn);
    case 6: return oz_kernel_tn<6>(tn);
    default: return oz_kernel_tn<7>(tn);
  }
}

}  // namespace

OzBuf oz_buf_alloc(int rows, int K, int smax, int nkb) {
  return oz_buf_alloc_raw(oz_plane_elems(rows, K, smax),
                          (size_t)((rows + kOzTileM - 1) / kOzTileM) * kOzTileM * std::max(nkb, 1));
}

OzBuf oz_buf_alloc_raw(size_t plane_elems, size_t exp_elems) {
  OzBuf b;
  b.cap = plane_elems;
  b.ecap = exp_elems;
  void* p = nullptr;
  if (cudaMalloc(&p, sizeof(uint16_t) * b.cap) != cudaSuccess) throw RihfError(RIHF_ERR_OOM, "cudaMalloc failed");
  b.planes = static_cast<uint16_t*>(p);
  if (cudaMalloc(&p, sizeof(int) * b.ecap) != cudaSuccess) {
    cudaFree(b.planes);
    throw RihfError(RIHF_ERR_OOM, "cudaMalloc failed");
  }
  b.exps = static_cast<int*>(p);
  return b;
}

void oz_buf_free(OzBuf& b) {
  if (b.planes) cudaFree(b.planes);
  if (b.exps) cudaFree(b.exps);
  b = OzBuf();
}

OzOperand oz_slice(const LaCtx& la, const double* X, int rows, int K, long long s_r, long long s_k1,
                   long long s_k2, int KR, int smax, int kb_chunks, const OzBuf& buf, int RR, long long s_r2,
                   int packed_n) {
  if (rows <= 0 || K <= 0 || smax < 1 || smax > kOzMaxDigits || KR <= 0)
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_slice: bad arguments");
  uint16_t* planes = buf.planes;
  int* exps = buf.exps;
  OzOperand op;
  op.planes = planes;
  op.exps = exps;
  op.rows = rows;
  op.rows_pad = (rows + kOzTileM - 1) / kOzTileM * kOzTileM;
  op.kchunks = (K + kOzChunk - 1) / kOzChunk;
  op.smax = smax;
  op.kb_chunks = (kb_chunks <= 0 || kb_chunks > op.kchunks) ? op.kchunks : kb_chunks;
  op.nkb = (op.kchunks + op.kb_chunks - 1) / op.kb_chunks;
  if (oz_plane_elems(rows, K, smax) > buf.cap || (size_t)op.rows_pad * op.nkb > buf.ecap)
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_slice: digit-plane buffer too small");
  if (op.kchunks > 65535) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_slice: K too long");
  if (packed_n > 0 && (K != packed_n || rows % packed_n != 0))
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_slice: packed rows must be whole matrices");
  OzSrc S{X, rows, K, s_r, s_k1, s_k2, KR, RR, s_r2, packed_n, 0};
  auto even = [](long long v) { return v % 2 == 0; };
  S.vec = packed_n == 0 && s_k1 == 1 && K % 8 == 0 && (KR >= K || (KR % 8 == 0 && even(s_k2))) && even(s_r) &&
          (RR <= 0 || even(s_r2)) && (uintptr_t)X % 16 == 0;
  int slots = 1;   // warps that share a row's chunks
  while (slots < kOzThreads / 32 && slots < op.kb_chunks) slots *= 2;
  const dim3 grid(op.rows_pad / (8 * (kOzThreads / 32 / slots)), op.nkb);
  oz_slice_kernel<<<grid, kOzThreads, 0, la.stream>>>(S, op.kchunks, smax, op.kb_chunks, op.nkb, slots, exps, planes);
  RIHF_LAUNCH_CHECK();
  if (la.launches) *la.launches += 1;
  return op;
}

// Column tile of a GEMM that does not state one.  A tile's time grows with its
// columns, so while narrow tiles leave SMs idle they cost nothing: the narrowest
// of 16, 32 with at most one tile an SM (n = 384, 7 digits: 28 / 33 / 55 k clocks at
// 16 / 32 / 64; n = 192: 18 / 23 / 39 k).  Above that the operand loads of a tile
// are what repeats, and the widest is best (1024 x 12000, K = 256: 596 / 352 / 330 k),
// with 65..96 columns as two tiles of 48 (80 columns: 267 / 327 k at 48 / 64 and
// 7 digits, 176 / 200 k at 5).  No tile straddles a 128-row plane: the widths divide
// 128 or all tiles lie in the first one.
static int oz_column_tile(int M, int N, int nsplit, bool lower_only, int sms) {
  const long long rows = (long long)(M + kOzTileM - 1) / kOzTileM * nsplit;
  for (int tn : {16, 32}) {
    if (N <= tn) return tn;
    long long tiles = rows * ((N + tn - 1) / tn);
    if (lower_only) tiles = tiles / 2 + rows * (kOzTileM / tn) / 2;   // those on and below the diagonal
    if (tiles <= sms) return tn;
  }
  if (N <= kOzMaxTN) return (N + 15) / 16 * 16;
  return N <= 96 ? 48 : kOzMaxTN;
}

void oz_gemm(const LaCtx& la, const OzGemmArgs& g) {
  if (g.M <= 0 || g.N <= 0) return;
  const OzOperand &A = g.A, &B = g.B;
  if (g.s < 1 || g.s > kOzMaxDigits || g.s > A.smax || g.s > B.smax || A.kchunks != B.kchunks ||
      A.kb_chunks != B.kb_chunks || A.nkb != B.nkb || A.rows < g.M || B.rows < g.N)
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: operands do not match");
  if (A.kb_chunks > kMaxChunksPerBlock)
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: K block longer than the int64 accumulator allows");
  if (!g.atomic && A.nkb > 1) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: K blocks need atomic output");
  if (g.atomic && g.accumulate) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: atomic and accumulate");
  if (!la.sched) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: no work counter");
  OzTiling T;
  T.M = g.M;
  T.N = g.N;
  if (g.tn < 0 || g.tn % 16 || g.tn > kOzMaxTN ||
      (g.tn > 0 && g.N > g.tn && 128 % g.tn && (g.N + g.tn - 1) / g.tn * g.tn > 128))
    throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: bad column tile");
  const int sms = la.sms > 0 ? la.sms : 152;
  T.TN = g.tn > 0 ? g.tn : oz_column_tile(g.M, g.N, A.nkb, g.lower_only, sms);
  T.s = g.s;
  if (T.s * T.TN > kTmemCols) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: accumulators exceed TMEM");
  T.mtiles = (g.M + kOzTileM - 1) / kOzTileM;
  T.ntiles = (g.N + T.TN - 1) / T.TN;
  T.nsplit = A.nkb;
  const long long nitems = (long long)T.mtiles * T.ntiles * T.nsplit;
  if (nitems >= (1LL << 30)) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: too many tiles");
  T.nitems = (int)nitems;
  T.nfast = g.M > g.N ? 1 : 0;   // items next to each other share the larger operand's tile
  T.lower_only = g.lower_only ? 1 : 0;
  T.symcols = g.symcols;
  T.kb_chunks = A.kb_chunks;
  T.kchunks = A.kchunks;
  T.G = std::max(1, (1024 / T.s) / kOzChunk);
  T.stage_bytes = T.s * (kPlaneElems * 2 + T.TN * kOzChunk * 2);
  // what the drain warps need to add to C row by row
  const int stage_cols = T.TN % 32 == 0 ? 8 : 4;
  const int add_bytes = g.accumulate ? kDrainThreads * (stage_cols + 1) * 8 : 0;
  T.nst = std::min(kMaxStages, (kSmemMax - kBookBytes - 1024 - add_bytes) / T.stage_bytes);
  if (T.nst < 1) throw RihfError(RIHF_ERR_INVALID_ARG, "oz_gemm: stage exceeds shared memory");
  // a power of two goes into the integer result instead of an FP64 product
  int aexp = 0;
  const double amant = std::frexp(g.alpha, &aexp);
  const bool pow2 = std::fabs(amant) == 0.5;
  T.aexp = pow2 ? aexp - 1 : 0;
  T.aneg = pow2 && g.alpha < 0.0 ? 1 : 0;
  T.scale = pow2 ? 0 : 1;
  const int smem = std::max(kSmemMin, T.nst * T.stage_bytes + kBookBytes + 1024 + add_bytes);
  const OzKernel kernel = oz_kernel(T.s, T.TN);
  raise_smem_limit((const void*)kernel, kSmemMax);
  const int grid = (int)std::min<long long>(nitems, sms);
  kernel<<<grid, kGemmThreads, smem, la.stream>>>(A, B, T, g.alpha, g.C, g.MR, g.cs_m1, g.cs_m2, g.cs_n,
                                                          g.atomic ? 1 : (g.accumulate ? 2 : 0), la.flag, la.sched);
  RIHF_LAUNCH_CHECK();
  if (la.launches) *la.launches += 1;
}

}  // namespace rihf
