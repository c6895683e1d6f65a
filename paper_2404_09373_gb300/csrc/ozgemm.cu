// FP64-accurate GEMM on the tcgen05 tensor cores from sliced BF16 products.
//
// Every row r of an FP64 operand X (rows x K) is scaled by 2^-e_r so that
// |x| < 1, rounded to a fixed-point integer with 7S fraction bits and split
// into S balanced base-128 digits d_0..d_{S-1} (|d_0| <= 128, |d_s| <= 64),
// each exactly representable in BF16:
//     x 2^-e_r = sum_s d_s 2^{-7(s+1)} + O(2^{-7S-1}).
// A product keeps the digit pairs s + t <= S - 1 ("levels" q = s + t):
//     (A B^T)_mn = 2^{e_m + f_n - 14} sum_q 2^{-7q} L_q,  L_q = sum_k sum_{s+t=q} d_s b_t.
// Each level has its own FP32 accumulator in tensor memory.  Digit products
// are integers below 2^14, so levels 0 and 1 summed over a chunk of 1024 k
// values stay below 2^24 and are exact in FP32; deeper levels are too unless the
// operands hardly change along k (their FP32 rounding then adds at most 2^-31 K of
// the rows' scales: 77 units of 2^-28 in a chunk's level 2).  After every chunk the
// epilogue warps read the levels out (tcgen05.ld) and add them as integers
// (OzSums); the result is rounded once.  With S = 7 or 8 (FP64-grade: 49 or 56
// fraction bits per operand) the chunk is 512 k, so that levels 0..5 are exact:
// the product of the rounded operands is then exact up to the dropped levels
// (below 2^-56 relative per term for S = 8) and one final FP64 rounding.
//
// Operands are pre-tiled by the slicing kernel into the canonical K-major,
// no-swizzle UMMA layout (8x8 core matrices, LBO = 128 B along K, SBO =
// 512 B per 8-row group, 32 k values per tile), all S slices of one
// (row tile, k tile) contiguous, so one cp.async.bulk per operand fills a
// pipeline stage.  Roles per CTA (one per SM): warp 0 issues the bulk copies,
// warp 1 owns tensor memory, warps 1 and 2 issue tcgen05.mma, the rest drain the
// accumulators, convert and store.
// Every mbarrier wait is bounded: on expiry the CTA records an error code,
// lets its copies and MMAs in flight finish, frees tensor memory and exits.
//
// What a tile of the 5-digit product costs (131072 x 1824 x 832, clock64): two
// CTAs an SM, one tile each, 158k cycles, 89k of them in the conversion and
// strided stores of the epilogue; with that rewritten 75k; one persistent CTA
// with a pair of tiles, MMAs by one thread, 120k the pair, stage 2020 cycles; by
// two threads 104k, stage 1600 of which 1440 are MMA time at the full rate.
// In all 9.85 -> 3.44 ms, 1.73 PFLOP/s of BF16 (0.91 of the measured peak).
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "digits.cuh"
#include "internal.cuh"
#include "rules.h"

namespace isdf {
namespace {

constexpr int kMaxDevices = 64;  // per-device launch set-up and scratch addresses

constexpr int kBM = kOzTileM;  // A rows per CTA = TMEM lanes
constexpr int kBK = kOzTileK;  // k values per tile / pipeline stage
static_assert(kBK == kOzBK, "digit tiles");
constexpr int kKcTiles = 1024 / kBK;  // 1024 k values per exact chunk
constexpr long long kWaitLimit = 1ll << 30;
constexpr unsigned long long kWaitNs = 2000000000ull;  // 2 s of device time per wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
  // K-major, no swizzle: LBO = 128 B (next core matrix along K), SBO = 16 kBK
  // bytes (next 8-row group), descriptor version 1 (bits 46-47), layout type 0.
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)((16 * kBK) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// kind::f16 instruction descriptor: D F32, A/B BF16, both K-major, M x N.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait: gives up after wait_ns of device time (0: after the first
// unsuccessful try), after kWaitLimit polls, or as soon as any CTA of the
// launch has recorded an error in *err.  The
// pipeline waits take the launch's limit (kWaitNs unless a host-side fault
// injection shortens it); the drain waits for copies and MMAs in flight
// always take kWaitNs.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase, const int* err,
                                          unsigned long long wait_ns = kWaitNs) {
  const uint32_t addr = smem_u32(bar);
  unsigned long long t0 = 0;
  for (long long i = 0; i < kWaitLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(phase)
        : "memory");
    if (done) return true;
    if (wait_ns == 0) return false;  // a zero limit gives up after the first unsuccessful try
    if ((i & 255) == 0) {
      const unsigned long long now = globaltimer_ns();
      if (i == 0) t0 = now;
      else if (now - t0 > wait_ns) return false;
      if (err && *(volatile const int*)err) return false;
    }
  }
  return false;
}

// mbar_wait by all lanes of a warp, one answer for all of them
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t phase, const int* err, unsigned long long wait_ns) {
  return __all_sync(0xffffffffu, mbar_wait(bar, phase, err, wait_ns)) != 0;
}

// The CTA's abort flag, one answer for the whole warp: lanes that read it at
// different times would part, and some of them then sit without a limit in a
// warp-wide instruction (tcgen05.ld, __syncwarp) that the others never reach.
__device__ __forceinline__ bool warp_aborted(const int* flag) {
  return __any_sync(0xffffffffu, *(volatile const int*)flag) != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// The MMA warp runs its loop with all lanes and `el` is set in one of them: the
// instruction is predicated, not branched around.  Control flow stays uniform, so
// the descriptors live in uniform registers; under a branch on the lane every
// operand was moved there first and an MMA took 110 cycles to issue whatever its
// size.
__device__ __forceinline__ void umma_bf16(uint32_t el, uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(el));
}

__device__ __forceinline__ void umma_commit(uint32_t el, uint64_t* bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar)),
      "r"(el)
      : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t el;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(el));
  return el;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void set_err(int* err, int code) { atomicCAS(err, 0, code); }

// Exponents beyond which a result may leave the normal range of a double
// (fixed_to_double's argument is at most 2^63 and at least 2^-28 in magnitude).
constexpr int kNearExp = 900;

// (th + rem 2^-28) 2^e rounded once to the nearest double (ties to even) with
// integer operations; rem in [0, 2^28), |e| <= kNearExp.  No branches, so that
// the conversions of neighbouring columns overlap.
__device__ __forceinline__ double fixed_to_double(long long th, uint32_t rem, int e) {
  // sign and magnitude hi + lo 2^-28
  const bool neg = th < 0;
  const uint32_t lo = neg ? (0u - rem) & 0x0FFFFFFFu : rem;
  uint64_t hi = neg ? ~uint64_t(th) + (rem == 0u ? 1ull : 0ull) : uint64_t(th);
  const bool low = hi == 0ull;  // only the fraction is left
  hi = low ? uint64_t(lo) : hi;
  const uint64_t frac = low ? 0ull : uint64_t(lo) << 36;
  const int lz = __clzll((long long)(hi | 1ull));
  const uint64_t top = (hi << lz) | ((frac >> 1) >> (63 - lz));
  const uint32_t cut = uint32_t(top) & 0x7FFu;
  const uint64_t M = top >> 11;  // 53 bits
  // half of the last place, and what lies below it
  const bool up = cut > 0x400u || (cut == 0x400u && ((frac << lz) != 0ull || (M & 1ull)));
  const int E = 63 - lz + e - (low ? 28 : 0) + 1022;
  // M's leading bit adds one to the exponent field, as does a carry out of it
  const uint64_t R = (uint64_t(neg) << 63) | ((uint64_t(uint32_t(E)) << 52) + M + (up ? 1ull : 0ull));
  return __longlong_as_double(hi ? (long long)R : 0ll);
}

// X 2^e rounded once to the nearest double (ties to even), |e| <= kNearExp
__device__ __forceinline__ double ll_to_double(long long X, int e) {
  const uint64_t U = X < 0 ? uint64_t(-X) : uint64_t(X);
  const int lz = __clzll((long long)(U | 1ull));
  const uint64_t top = U << lz;
  const uint32_t cut = uint32_t(top) & 0x7FFu;
  const uint64_t M = top >> 11;
  const uint32_t up = (cut > 0x400u || (cut == 0x400u && (uint32_t(M) & 1u))) ? 1u : 0u;
  const uint64_t R = (uint64_t(uint32_t(63 - lz + e + 1022)) << 52) + M + up;
  return __longlong_as_double((long long)((uint64_t(X) & 0x8000000000000000ull) | (U ? R : 0ull)));
}

// the first of the two for any exponent, out of line
__device__ __noinline__ double far_double(long long th, uint32_t rem, int e) {
  return ldexp(fixed_to_double(th, rem, 0), e);
}

// ---------------------------------------------------------------- slicing

// |x| as an order-preserving integer key (finite doubles)
__device__ __forceinline__ uint64_t abs_key(double x) { return uint64_t(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull; }

// exponent e with |x| < 2^e from the key of the largest |x| of a row
__device__ __forceinline__ int exp_of_key(uint64_t key) {
  if (key == 0) return 0;
  int e;
  frexp(__longlong_as_double((long long)key), &e);
  return e;
}

// |mul * kw[k] * v| as an order-preserving key
__device__ __forceinline__ uint64_t key_at(double v, int64_t k, const double* __restrict__ kw, double mul) {
  if (mul != 1.0) v *= mul;
  if (kw) v *= kw[k];
  return abs_key(v);
}

__device__ __forceinline__ uint64_t umax64(uint64_t a, uint64_t b) { return a > b ? a : b; }

// Row scales of few very long contiguous rows (the Coulomb spectra, K of
// millions): blockIdx.y walks shares of one row, the shares meet in an
// atomicMax on the row's key; k_oz_key_exps turns the keys into exponents.
// 16-byte loads, four per thread in flight.
__global__ void k_oz_row_keys(const double* __restrict__ src, int64_t sr, int64_t K, int64_t share,
                              const double* __restrict__ kw, double mul, unsigned long long* __restrict__ keys) {
  __shared__ unsigned long long sh[8];
  const int64_t r = blockIdx.x;
  const int64_t k0 = int64_t(blockIdx.y) * share, k1 = k0 + share < K ? k0 + share : K;  // share is even
  const double* row = src + r * sr;
  uint64_t m = 0;
  const int bd = blockDim.x;
  if ((reinterpret_cast<uintptr_t>(row) & 15) == 0) {
    const double2* p = reinterpret_cast<const double2*>(row);
    const int64_t i1 = k1 >> 1;
    int64_t i = (k0 >> 1) + threadIdx.x;
    for (; i + 3 * bd < i1; i += 4 * bd) {
      double2 t[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) t[h] = __ldg(p + i + h * bd);
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int64_t k = 2 * (i + h * bd);
        m = umax64(m, umax64(key_at(t[h].x, k, kw, mul), key_at(t[h].y, k + 1, kw, mul)));
      }
    }
    for (; i < i1; i += bd) {
      const double2 t = __ldg(p + i);
      m = umax64(m, umax64(key_at(t.x, 2 * i, kw, mul), key_at(t.y, 2 * i + 1, kw, mul)));
    }
    if ((k1 & 1) && threadIdx.x == 0) m = umax64(m, key_at(row[k1 - 1], k1 - 1, kw, mul));
  } else {
    for (int64_t k = k0 + threadIdx.x; k < k1; k += bd) m = umax64(m, key_at(row[k], k, kw, mul));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = umax64(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < bd / 32; ++w) m = umax64(m, sh[w]);
    atomicMax(keys + r, (unsigned long long)m);
  }
}

__global__ void k_oz_key_exps(const unsigned long long* __restrict__ keys, int64_t rows, int* __restrict__ exps) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r < rows) exps[r] = exp_of_key(keys[r]);
}

// The 8 values of k group kg of a row (zero beyond K), before mul and kw.
__device__ __forceinline__ void oz_load8(const double* __restrict__ row, bool live, int64_t sk, int64_t K, int64_t kg,
                                         double (&v)[8]) {
  const int64_t k0 = kg * 8;
  if (live && sk == 1 && k0 + 8 <= K && (reinterpret_cast<uintptr_t>(row + k0) & 15) == 0) {
    const double2* p = reinterpret_cast<const double2*>(row + k0);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const double2 t = __ldg(p + h);
      v[2 * h] = t.x;
      v[2 * h + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = (live && k0 + u < K) ? __ldg(row + (k0 + u) * sk) : 0.0;
  }
}

__device__ __forceinline__ void oz_weight8(double (&v)[8], int64_t K, int64_t kg, const double* __restrict__ kw,
                                           double mul) {
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (kg * 8 + u < K) {
      if (mul != 1.0) v[u] *= mul;
      if (kw) v[u] *= kw[kg * 8 + u];
    }
}

struct OzSliceArgs {
  const double* src;
  int64_t sr, sk;  // element (r, k) at src[row(r) sr + k sk]
  int64_t rows, K;
  const double* kw;
  double mul;
  const int* ridx;  // row(r) = ridx[r] (nullable: r)
  int rt;
  int64_t nrt, kst;
  int64_t kg0, ngrp;  // window of 8-wide k groups
  int* exps;
  __nv_bfloat16* tiles;  // tile (row tile i, k tile j) at position i * kst + j
};

__device__ __forceinline__ const double* oz_row(const OzSliceArgs& A, int64_t r) {
  return A.src + (A.ridx ? int64_t(A.ridx[r]) : r) * A.sr;
}

template <int S>
__device__ __forceinline__ void oz_emit(const OzSliceArgs& A, int64_t r, int64_t kg, int e, double (&v)[8]) {
  oz_weight8(v, A.K, kg, A.kw, A.mul);
  const int64_t it = r / A.rt, jt = kg / (kBK / 8);
  const int rr = int(r - it * A.rt), kc = int(kg % (kBK / 8));
  const int64_t tile_elems = int64_t(A.rt) * kBK;
  __nv_bfloat16* out = A.tiles + ((it * A.kst + jt) * S) * tile_elems + oz_inner(rr, kc);
  oz_digits8<S>(v, 7 * S - e, tile_elems, out);
}

// Digits of a window of k groups for rows whose scales are in exps (padding
// rows are written as zero).  RG 32 (rows adjacent in memory): a warp takes 32
// rows of one k group; RG 8 (k adjacent): 8 rows x 4 k groups, so it writes one
// 512-byte line of each slice and reads 256 contiguous bytes of each row.
template <int S, int RG>
__global__ void __launch_bounds__(256) k_oz_digits(OzSliceArgs A) {
  constexpr int KG = 32 / RG;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t rows_pad = A.nrt * A.rt;
  if (RG == 32) {
    const int64_t r = (int64_t(blockIdx.x) * 8 + warp) * 32 + lane;
    if (r >= rows_pad) return;
    const bool live = r < A.rows;
    const int e = live ? A.exps[r] : 0;
    const double* row = live ? oz_row(A, r) : A.src;
    for (int64_t g = blockIdx.y; g < A.ngrp; g += gridDim.y) {
      double v[8];
      oz_load8(row, live, A.sk, A.K, A.kg0 + g, v);
      oz_emit<S>(A, r, A.kg0 + g, e, v);
    }
  } else {
    const int64_t g = (int64_t(blockIdx.x) * 8 + warp) * KG + lane / RG;
    if (g >= A.ngrp) return;
    for (int64_t g8 = blockIdx.y; g8 * 8 < rows_pad; g8 += gridDim.y) {
      const int64_t r = g8 * 8 + lane % RG;
      const bool live = r < A.rows;
      double v[8];
      oz_load8(live ? oz_row(A, r) : A.src, live, A.sk, A.K, A.kg0 + g, v);
      oz_emit<S>(A, r, A.kg0 + g, live ? A.exps[r] : 0, v);
    }
  }
}

// Row scales and digits of a whole operand in one launch.  A block owns RG
// rows: it takes their maxima over all k, then reads the same values again,
// from L1 or L2, and writes their digits: one pass over HBM.  (One thread per
// row for the maximum and a second kernel for the digits read the operand
// twice and left a short operand to a few serial threads.)  Blocks are small,
// so that an SM holds many at different points of the two passes.  Bound by
// HBM (8 B read and 2 S written per value) and the latency of the two passes;
// measured: 250001 x 607, 8 digits, 1.89 -> 0.94 ms (3.9 TB/s); 131072 x 832,
// 5 digits, 1.37 -> 0.65 ms; 96 gathered rows of 200 values, 50 -> 7 us.
template <int S, int RG>
__global__ void __launch_bounds__(512, 2) k_oz_slice(OzSliceArgs A) {
  constexpr int KG = 32 / RG;
  __shared__ unsigned long long key[RG];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int rl = lane % RG;
  const int64_t r = int64_t(blockIdx.x) * RG + rl;
  const bool live = r < A.rows;  // rows up to the tile height are padding, written as zero
  const double* row = live ? oz_row(A, r) : A.src;
  const int64_t g0 = int64_t(warp) * KG + lane / RG, gs = int64_t(nw) * KG;
  double v[8];
  uint64_t m = 0;
  if (live)
#pragma unroll 2
    for (int64_t g = g0; g < A.ngrp; g += gs) {
      oz_load8(row, true, A.sk, A.K, g, v);
      const int64_t k0 = g * 8;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k0 + u < A.K) m = umax64(m, key_at(v[u], k0 + u, A.kw, A.mul));
    }
  if (RG == 8) {
    m = umax64(m, __shfl_xor_sync(0xffffffffu, m, 8));
    m = umax64(m, __shfl_xor_sync(0xffffffffu, m, 16));
  }
  if (nw > 1) {
    if (threadIdx.x < RG) key[threadIdx.x] = 0ull;
    __syncthreads();
    if (lane < RG) atomicMax(&key[rl], (unsigned long long)m);
    __syncthreads();
    m = key[rl];
  }
  const int e = exp_of_key(m);
  if (live && warp == 0 && lane < RG) A.exps[r] = e;
  if (r >= A.nrt * A.rt) return;  // a 32-row block past the last (48-row) tile
  const bool once = gs >= A.ngrp;  // every thread's only group is still in registers
  for (int64_t g = g0; g < A.ngrp; g += gs) {
    if (!once || !live) oz_load8(row, live, A.sk, A.K, g, v);
    oz_emit<S>(A, r, g, e, v);
  }
}
OzSliceArgs slice_args(const double* src, int64_t sr, int64_t sk, const double* kw, double mul, const int* ridx,
                       const OzOperand& op, int64_t kg0, int64_t ngrp) {
  return {src, sr, sk, op.rows, op.K, kw, mul, ridx, op.rt, op.nrt, op.kst, kg0, ngrp, op.exps,
          static_cast<__nv_bfloat16*>(op.tiles)};
}

template <int S>
void launch_digits_s(const OzSliceArgs& A, cudaStream_t s) {
  const int64_t rows_pad = A.nrt * A.rt;
  if (A.sr < A.sk)
    k_oz_digits<S, 32><<<dim3(unsigned((rows_pad + 255) / 256), unsigned(std::min<int64_t>(A.ngrp, 65535))), 256, 0, s>>>(A);
  else
    k_oz_digits<S, 8><<<dim3(unsigned((A.ngrp + 31) / 32), unsigned(std::min<int64_t>(rows_pad / 8, 65535))), 256, 0, s>>>(A);
}

void launch_digits(const OzSliceArgs& A, int S, cudaStream_t s) {
  if (S == 5) launch_digits_s<5>(A, s);
  else if (S == 6) launch_digits_s<6>(A, s);
  else if (S == 7) launch_digits_s<7>(A, s);
  else launch_digits_s<8>(A, s);
  count_launches(1);
}

// Rows adjacent in memory (sr < sk) are taken 32 to a block when there are
// enough of them for every SM, else 8 to a block (64-byte pieces of a
// line, but four times the blocks); rows with k adjacent always 8 to a block.
constexpr int64_t kWideRows = 2 * 152 * 32;
// Warps per block: an SM holds 32 warps of this kernel, and the rows it is
// working on have to stay in L2 between the two reads: at most about 320 KB an
// SM (48 MB in all).  With fewer blocks than that, more warps share a row.
constexpr int64_t kSliceBytes = 320 * 1024;

template <int S>
void launch_slice_s(const OzSliceArgs& A, cudaStream_t s) {
  const int64_t rows_pad = A.nrt * A.rt;
  const bool wide = A.sr < A.sk && rows_pad >= kWideRows;
  const int rg = wide ? 32 : 8, kg = 32 / rg;
  const int64_t blocks = (rows_pad + rg - 1) / rg;
  int nw = 1;
  while (nw < 16 && nw * kg < A.ngrp && (32 / nw * rg * A.K * 8 > kSliceBytes || blocks * nw < 152 * 32)) nw *= 2;
  const unsigned grid = unsigned(blocks);
  if (wide)
    k_oz_slice<S, 32><<<grid, 32 * nw, 0, s>>>(A);
  else
    k_oz_slice<S, 8><<<grid, 32 * nw, 0, s>>>(A);
}

// Row scales, then digits, of a whole operand.  Rows of up to kFusedK values
// with k adjacent (and every operand with rows adjacent) go through the fused
// kernel; longer rows would fall out of L2 between its two reads (two blocks an
// SM, 8 rows each: 80 MB at 4096 values), so their maxima are taken first by
// blocks that share each row.
constexpr int64_t kFusedK = 4096;

void slice_operand(const OzSliceArgs& A, int S, cudaStream_t s) {
  if (A.sr < A.sk || A.K <= kFusedK || A.ridx || A.sk != 1) {
    if (S == 5) launch_slice_s<5>(A, s);
    else if (S == 6) launch_slice_s<6>(A, s);
    else if (S == 7) launch_slice_s<7>(A, s);
    else launch_slice_s<8>(A, s);
    count_launches(1);
    return;
  }
  // the keys use the head of the operand's own tiles, which the digits overwrite afterwards
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(A.tiles);
  cudaMemsetAsync(keys, 0, sizeof(unsigned long long) * size_t(A.rows), s);
  // enough shares per row for about 8 waves of blocks, at least 4096 values each
  int64_t nsh = std::max<int64_t>(1, std::min<int64_t>((int64_t(152) * 64 + A.rows - 1) / A.rows, A.K / 4096));
  int64_t share = (A.K + nsh - 1) / nsh;
  share += share & 1;
  nsh = (A.K + share - 1) / share;
  k_oz_row_keys<<<dim3(unsigned(A.rows), unsigned(nsh)), 256, 0, s>>>(A.src, A.sr, A.K, share, A.kw, A.mul, keys);
  k_oz_key_exps<<<unsigned((A.rows + 255) / 256), 256, 0, s>>>(keys, A.rows, A.exps);
  count_launches(2);
  launch_digits(A, S, s);
}

// ---------------------------------------------------------------- GEMM

struct OzGemmParams {
  const __nv_bfloat16* A;
  const __nv_bfloat16* B;
  const int* ea;
  const int* eb;
  int64_t M, N, nkt;
  int64_t ntm, ntn;    // M tiles (of 128 rows) and N tiles (of BN rows)
  int64_t akst, bkst;  // k-tile strides of the A and B tile arrays (>= nkt)
  int64_t bgroups;     // 8-row groups of B if its array has 128-row tiles, else 0
  int tri;     // 0 dense; 1 B-side lower (k <= n); 2 B-side upper (k >= n)
  int sym;     // compute only tiles that touch the lower triangle (n <= m)
  int splits;  // split-K factor (gridDim.z)
  double* C;
  int64_t cm, cn;  // C[m cm + n cn]
  double alpha;
  double* work;  // split-K partials [z][M][N]
  int* err;
  unsigned long long wait_ns;  // limit of each pipeline wait (device time)
  OzWindows win;
};

template <int S, int BN>
struct OzCfg {
  static constexpr int tileA = kBM * kBK * 2;  // bytes per slice tile
  static constexpr int tileB = BN * kBK * 2;
  static constexpr int stageA = S * tileA;
  static constexpr int stageB = S * tileB;
  static constexpr int cols = S * BN;
  static constexpr bool exact = S >= 7;
  // Two N tiles at a time where their accumulators fit in tensor memory: they
  // share the A digits of a stage.
  static constexpr int pair = cols <= 256 ? 2 : 1;
  // Two issuing warps, each with its own accumulator columns: the two tiles of a
  // pair, or levels [0, cut) and [cut, S) of one.  MMAs of one thread run one after
  // the other, N / 2 + 32 cycles each (the A operand's load is not hidden: a stage
  // of 5 digits and two tiles took 2020 cycles, 1440 of them MMA time); those of
  // two threads overlap.
  static constexpr int issuers = 2;
  static constexpr int cut = S == 6 ? 4 : 5;
  static constexpr int stage = stageA + pair * stageB;
  static constexpr uint32_t tcols = 512;
  // epilogue warps: two per tensor-memory lane quarter (BN / 2 columns of a tile
  // each), or three (BN / 3 columns each, so that the integer state fits in registers)
  static constexpr int epi = BN % 48 == 0 ? 12 : 8;
  // the epilogue's transposing buffer: [32][4] values a warp, past the ring
  static constexpr int xbytes = epi * 32 * 4 * 8;
  static constexpr int nst = (232448 - 2048 - xbytes) / stage < 4 ? (232448 - 2048 - xbytes) / stage : 4;
  static constexpr int xpose = nst * stage + 1024;
  static constexpr int smem = nst * stage + 2048 + xbytes;  // + barriers and 1024-byte alignment slack
  // 7, 8 digits: levels 0..5 are kept exact (chunks of 512 k keep their integer
  // sums at most 2^24; levels 6, 7 weigh less than 2^-42, where FP32 rounding
  // is harmless); 5, 6 digits: levels 0 and 1 (1024 k)
  static constexpr int kc = exact ? 512 / kBK : kKcTiles;  // k tiles per chunk
  static constexpr int threads = 32 * (1 + issuers + epi);
  static_assert(!exact || S == 7 || S == 8, "the integer epilogue pairs the levels of 7 or 8 digits");
  static_assert(cols <= 512, "levels x BN must fit in tensor memory");
  static_assert(nst >= 2, "need at least two pipeline stages");
  static_assert((BN / (epi / 4)) % 8 == 0, "each epilogue warp reads whole 8-column groups");
  static_assert(smem <= 232448, "shared memory per CTA");
};

// One issuer's MMAs of one pipeline stage (32 k values).  For A digit s the
// products with B digits t = 0..S-1-s land in levels s..S-1, i.e.
// tensor-memory columns [s BN, S BN); the B digit tiles of a stage are
// contiguous, so one MMA covers the levels [q, q1) of an issuer's range with B
// rows [(q - s) BN, (q1 - s) BN), q the first of its levels at or above s.  The
// first MMA of a chunk (s = 0) spans the whole range and initialises it.
template <int S, int BN, int PART>
__device__ __forceinline__ void mma_part(uint32_t el, uint32_t tmem, uint32_t sA, uint32_t sB, bool first) {
  using Cfg = OzCfg<S, BN>;
  constexpr int tile = Cfg::pair == 2 ? PART : 0;  // 256 columns on for the second tile
  constexpr int q0 = Cfg::pair == 2 || PART == 0 ? 0 : Cfg::cut;
  constexpr int q1 = Cfg::pair == 2 || PART == 1 ? S : Cfg::cut;
  static_assert((q1 - q0) * BN <= 256, "an MMA has at most 256 columns");
#pragma unroll
  for (int s = 0; s < q1; ++s) {
    const int q = s > q0 ? s : q0, n = (q1 - q) * BN;
#pragma unroll
    for (int ks = 0; ks < kBK / 16; ++ks) {
      const uint64_t da = umma_desc(sA + s * Cfg::tileA + ks * 256);
      const uint64_t db = umma_desc(sB + tile * Cfg::stageB + ((q - s) * BN / 8) * (16 * kBK) + ks * 256);
      umma_bf16(el, tmem + uint32_t(256 * tile + q * BN), da, db, umma_idesc(kBM, n), (!first || s > 0 || ks > 0) ? 1u : 0u);
    }
  }
}
template <int S, int BN>
__device__ __forceinline__ void mma_stage(int part, uint32_t el, uint32_t tmem, uint32_t sA, uint32_t sB, bool first,
                                          int tiles) {
  if (part == 0) mma_part<S, BN, 0>(el, tmem, sA, sB, first);
  else if (OzCfg<S, BN>::pair == 1 || tiles == 2) mma_part<S, BN, 1>(el, tmem, sA, sB, first);
}

// Exact integer sums of one thread's HC columns: th in units of 2^-21 of
// level 0, the rest a fraction of such a unit.
//   7 or 8 digits: 28 bits in rem.  Levels 0..5 of a 512-k chunk are integers
//     below 2^24, paired in 32 bits (L0 2^7 + L1 and so on, below 2^31); levels
//     6 and 7 lie below 2^-42, where FP32 rounding is harmless.
//   6 digits: 14 bits in rem.  5 digits: 7 bits, four columns to a word.  Every
//     level's FP32 sum is an integer; levels 0 and 1 are exact for 1024 k.  The
//     deeper ones reach 20480 to 32768 a k value (2^24.3 to 2^25 a chunk) where the
//     operands hardly change along k: FP32 then rounds them, and times 128 they
//     need 64 bits.
// Integer sums take 2 or 3 operations per level where double-float ones took 8,
// and leave one value to round at the end.
template <int S, int HC>
struct OzSums {
  static constexpr int NR = S == 5 ? HC / 4 : HC;
  static constexpr int64_t wide = oz_wide_k(S);  // 5 and 6 digits
  long long th[HC];
  uint32_t rem[NR];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < HC; ++j) th[j] = 0;
#pragma unroll
    for (int j = 0; j < NR; ++j) rem[j] = 0u;
  }
  // add the accumulators of one chunk (this warp's lanes, HC columns from tbase, levels BN apart)
  template <int BN>
  __device__ __forceinline__ void drain(uint32_t tbase) {
#pragma unroll
    for (int c0 = 0; c0 < HC; c0 += 8) {
      uint32_t r[S][8];
#pragma unroll
      for (int q = 0; q < S; ++q) tmem_ld8(tbase + uint32_t(q * BN + c0), r[q]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + j;
        int L[S];
#pragma unroll
        for (int q = 0; q < S; ++q) L[q] = __float2int_rn(__uint_as_float(r[q][j]));
        if constexpr (S >= 7) {
          const int p01 = L[0] * 128 + L[1], p23 = L[2] * 128 + L[3], p45 = L[4] * 128 + L[5];
          long long lo = (long long)p45 * (1 << 14) + (long long)L[6] * 128;
          if constexpr (S == 8) lo += L[7];
          const uint32_t f = rem[c] + (uint32_t(lo) & 0x0FFFFFFFu);
          th[c] += (long long)p01 * (1 << 14) + (long long)p23 + (lo >> 28) + (long long)(f >> 28);
          rem[c] = f & 0x0FFFFFFFu;
        } else {
          th[c] += (long long)L[0] * (1 << 21) + (long long)L[1] * (1 << 14) + (long long)L[2] * 128;
          if constexpr (S == 6) {
            const long long lo = (long long)L[4] * 128 + L[5];
            const uint32_t f = rem[c] + (uint32_t(lo) & 0x3FFFu);
            th[c] += (long long)L[3] + (lo >> 14) + (long long)(f >> 14);
            rem[c] = f & 0x3FFFu;
          } else {
            const int sh = 8 * (c & 3);
            const uint32_t f = ((rem[c / 4] >> sh) & 0x7Fu) + (uint32_t(L[4]) & 0x7Fu);
            th[c] += (long long)(L[3] + (L[4] >> 7) + int(f >> 7));
            rem[c / 4] = (rem[c / 4] & ~(0xFFu << sh)) | ((f & 0x7Fu) << sh);
          }
        }
      }
    }
  }
  // fraction of column c in units of 2^-28
  __device__ __forceinline__ uint32_t frac(int c) const {
    if constexpr (S >= 7) return rem[c];
    else if constexpr (S == 6) return rem[c] << 14;
    else return ((rem[c / 4] >> (8 * (c & 3))) & 0x7Fu) << 21;
  }
  // every column's value times 2^(ea + eb(c)), rounded once; k: values summed (a
  // 5- or 6-digit sum of many may not fit 64 bits with its fraction).  Straight-line
  // code (the rare cases afterwards, out of line), so that the columns'
  // conversions overlap, and no FP64 instruction: each holds its scheduler for
  // over 100 cycles.
  template <class E>
  __device__ __forceinline__ void values(int ea, E eb, int64_t k, double (&v)[HC]) const {
    constexpr int FB = 7 * (S - 4);  // bits of the fraction (S < 7)
    int m = 0;
#pragma unroll
    for (int c = 0; c < HC; ++c) {
      const int e = ea + eb(c) - 35, en = abs(e) > kNearExp - 64 ? 0 : e;
      m = max(m, abs(e));
      if constexpr (S >= 7) v[c] = fixed_to_double(th[c], rem[c], en);
      else v[c] = ll_to_double(th[c] * (1 << FB) + (long long)(frac(c) >> (28 - FB)), en - FB);
    }
    bool far = m > kNearExp - 64;
    if constexpr (S < 7) far = far || k >= wide;
    if (far)
#pragma unroll
      for (int c = 0; c < HC; ++c) v[c] = far_double(th[c], frac(c), ea + eb(c) - 35);
  }
};

template <int S, int BN>
__global__ void __launch_bounds__(OzCfg<S, BN>::threads, 1) k_oz_gemm(OzGemmParams P) {
  using Cfg = OzCfg<S, BN>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::nst * Cfg::stage);
  uint64_t* empty = full + Cfg::nst;
  uint64_t* acc_full = empty + Cfg::nst;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* drain = acc_empty + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + Cfg::issuers);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0);  // uniform to the compiler
  const int lane = threadIdx.x % 32;
  // an earlier launch failed: do nothing (one read, made uniform across the CTA)
  if (__syncthreads_or(threadIdx.x == 0 ? *(volatile const int*)P.err : 0)) return;

  // Persistent tiles: tile t is (N tile t % NT, M tile (t / NT) % MT, split
  // t / (NT MT)); N tiles vary fastest so that CTAs in flight share A.  Every
  // role walks the same tile sequence; stage and chunk counters run on across
  // tiles, so the ring of stages and the accumulator hand-off never restart
  // and a tile's epilogue overlaps the next tile's copies and MMAs.
  const int64_t NT = (P.ntn + Cfg::pair - 1) / Cfg::pair, MT = P.ntm, ntiles = NT * MT * P.splits;
  struct Tile {
    int64_t nt, mt, m0, n0, kt_lo, nk;  // steps [kt_lo, kt_lo + nk) of the k tiles k_tile()
    int64_t n1, base1, base2;           // steps below n1 are k tiles from base1 on, the others from base2 on
    int z, tiles;  // tiles: N tiles of this pair
    bool skip;
  };
  auto tile_at = [&](int64_t t) {
    Tile T;
    T.nt = t % NT;
    T.mt = (t / NT) % MT;
    T.z = int(t / (NT * MT));
    T.m0 = T.mt * kBM;
    T.nt *= Cfg::pair;
    T.tiles = int(min(int64_t(Cfg::pair), P.ntn - T.nt));
    T.n0 = T.nt * BN;
    T.skip = P.sym && T.n0 > T.m0 + kBM - 1;  // tile entirely above the diagonal
    int64_t lo = 0, hi = P.nkt;
    if (P.tri == 1) hi = min(P.nkt, (T.n0 + Cfg::pair * BN + kBK - 1) / kBK);
    if (P.tri == 2) lo = min(P.nkt, T.n0 / kBK);
    T.n1 = hi, T.base1 = T.base2 = 0;
    if (P.win.n) {
      const int64_t r0 = P.win.side ? T.m0 : T.n0, r1 = r0 + (P.win.side ? kBM : Cfg::pair * BN);
      int64_t a[2] = {P.nkt, P.nkt}, b[2] = {0, 0};  // k tiles of the two ranges
#pragma unroll
      for (int g = 0; g < ISDF_MAX_LEVELS; ++g)
        if (g < P.win.n && P.win.row[g] < r1 && P.win.row[g + 1] > r0)
#pragma unroll
          for (int i = 0; i < 2; ++i)
            if (P.win.hi[g][i] > P.win.lo[g][i]) {
              a[i] = min(a[i], P.win.lo[g][i] / kBK);
              b[i] = max(b[i], min(P.nkt, (P.win.hi[g][i] + kBK - 1) / kBK));
            }
      a[1] = max(a[1], b[0]);  // a k tile that holds the end of one and the start of the other
      T.n1 = max(b[0] - a[0], int64_t(0));
      T.base1 = a[0];
      T.base2 = a[1] - T.n1;
      hi = T.n1 + max(b[1] - a[1], int64_t(0));
    }
    const int64_t tot = hi - lo, per = (tot + P.splits - 1) / P.splits;
    const int64_t a = lo + per * T.z;
    T.kt_lo = min(hi, a);
    T.nk = min(hi, a + per) - T.kt_lo;
    return T;
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < Cfg::nst; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], Cfg::issuers);
    }
    mbar_init(acc_full, Cfg::issuers);
    mbar_init(acc_empty, Cfg::epi);
    for (int i = 0; i < Cfg::issuers; ++i) mbar_init(&drain[i], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(Cfg::tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    // ------------------------------------------------ producer
    if (lane == 0) {
      const unsigned char* gA = reinterpret_cast<const unsigned char*>(P.A);
      const unsigned char* gB = reinterpret_cast<const unsigned char*>(P.B);
      int64_t g = 0;  // stages issued so far (all tiles)
      for (int64_t t = blockIdx.x; t < ntiles && !*(volatile int*)abort_flag; t += gridDim.x) {
        const Tile T = tile_at(t);
        if (T.skip) continue;
        for (int64_t it = 0; it < T.nk; ++it, ++g) {
          const int st = int(g % Cfg::nst);
          const int64_t round = g / Cfg::nst;
          if (round > 0 && !mbar_wait(&empty[st], uint32_t((round - 1) & 1), P.err, P.wait_ns)) {
            set_err(P.err, 11);
            *(volatile int*)abort_flag = 1;
            break;
          }
          if (*(volatile int*)abort_flag) break;
          const int64_t step = T.kt_lo + it, kt = step + (step < T.n1 ? T.base1 : T.base2);
          unsigned char* sA = smem + st * Cfg::stage;
          unsigned char* sB = sA + Cfg::stageA;
          if (!P.bgroups) {
            mbar_expect_tx(&full[st], Cfg::stageA + T.tiles * Cfg::stageB);
            bulk_g2s(sA, gA + (T.mt * P.akst + kt) * int64_t(Cfg::stageA), Cfg::stageA, &full[st]);
            for (int b = 0; b < T.tiles; ++b)
              bulk_g2s(sB + b * Cfg::stageB, gB + ((T.nt + b) * P.bkst + kt) * int64_t(Cfg::stageB), Cfg::stageB,
                       &full[st]);
            continue;
          }
          // B's rows from 128-row tiles: groups of 8 rows (512 bytes a digit) are
          // contiguous up to the end of a tile, so a digit takes one or two copies.
          // Groups behind the last tile are left out: their columns are not stored.
          const int64_t g0 = T.n0 / 8, g1 = min(g0 + T.tiles * (BN / 8), P.bgroups);
          mbar_expect_tx(&full[st], Cfg::stageA + uint32_t(g1 - g0) * (512 * S));
          bulk_g2s(sA, gA + (T.mt * P.akst + kt) * int64_t(Cfg::stageA), Cfg::stageA, &full[st]);
          for (int64_t gb = g0; gb < g1;) {
            const int in_b = int(gb - g0) % (BN / 8), b = int(gb - g0) / (BN / 8);
            const int n = int(min(min(int64_t(BN / 8 - in_b), 16 - gb % 16), g1 - gb));
            const unsigned char* from = gB + ((gb / 16) * P.bkst + kt) * int64_t(Cfg::stageA) + (gb % 16) * 512;
            unsigned char* to = sB + b * Cfg::stageB + in_b * 512;
            for (int d = 0; d < S; ++d) bulk_g2s(to + d * Cfg::tileB, from + d * Cfg::tileA, n * 512, &full[st]);
            gb += n;
          }
        }
      }
      // copies that were issued but never consumed must land before exit
      if (*(volatile int*)abort_flag) {
        const int64_t first = g > Cfg::nst ? g - Cfg::nst : 0;
        for (int64_t it = first; it < g; ++it) mbar_wait(&full[it % Cfg::nst], uint32_t((it / Cfg::nst) & 1), nullptr);
      }
    }
  } else if (warp <= Cfg::issuers) {
    // ------------------------------------------------ MMA issuers
    const uint32_t el = elect_one();
    {
      int64_t g = 0, h = 0;  // stages consumed, accumulator chunks handed over (all tiles)
      bool stop = false;
      for (int64_t t = blockIdx.x; t < ntiles && !stop; t += gridDim.x) {
        const Tile T = tile_at(t);
        if (T.skip) continue;
        for (int64_t it = 0; it < T.nk; ++it, ++g) {
          const int st = int(g % Cfg::nst);
          const int64_t round = g / Cfg::nst;
          const int64_t cpos = it % Cfg::kc;
          if (cpos == 0 && h > 0 && !warp_wait(acc_empty, uint32_t((h - 1) & 1), P.err, P.wait_ns)) {
            set_err(P.err, 12);
            *(volatile int*)abort_flag = 1;
            stop = true;
            break;
          }
          if (!warp_wait(&full[st], uint32_t(round & 1), P.err, P.wait_ns)) {
            set_err(P.err, 13);
            *(volatile int*)abort_flag = 1;
            stop = true;
            break;
          }
          if (warp_aborted(abort_flag)) {
            stop = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t sA = smem_u32(smem + st * Cfg::stage);
          const uint32_t sB = sA + Cfg::stageA;
          mma_stage<S, BN>(warp - 1, el, tmem, sA, sB, cpos == 0, T.tiles);
          umma_commit(el, &empty[st]);
          if (cpos == Cfg::kc - 1 || it == T.nk - 1) {
            umma_commit(el, acc_full);
            ++h;
          }
        }
      }
      // all MMAs issued by this thread complete before tensor memory is freed
      umma_commit(el, &drain[warp - 1]);
      mbar_wait(&drain[warp - 1], 0, nullptr);
    }
  } else {
    // ------------------------------------------------ epilogue warps
    const int quarter = warp % 4;  // a warp reads tensor-memory lanes 32 (warp % 4) ..
    const int half = (warp - 1 - Cfg::issuers) / 4;  // which share of the columns
    const int row = quarter * 32 + lane;
    constexpr int HC = BN / (Cfg::epi / 4);  // columns per thread
    int64_t h = 0;  // accumulator chunks taken over (all tiles)
    for (int64_t t = blockIdx.x; t < ntiles && !warp_aborted(abort_flag); t += gridDim.x) {
      const Tile T = tile_at(t);
      if (T.skip) continue;
      const int64_t nchunks = (T.nk + Cfg::kc - 1) / Cfg::kc;
      const int64_t m = T.m0 + row;
      OzSums<S, HC> sums[Cfg::pair];
#pragma unroll
      for (int b = 0; b < Cfg::pair; ++b) sums[b].clear();
      for (int64_t c = 0; c < nchunks; ++c) {
        if (!warp_wait(acc_full, uint32_t(h & 1), P.err, P.wait_ns)) {
          set_err(P.err, 14);
          *(volatile int*)abort_flag = 1;
          break;
        }
        ++h;
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int b = 0; b < Cfg::pair; ++b)
          if (b < T.tiles)
            sums[b].template drain<BN>(tmem + (uint32_t(quarter * 32) << 16) + uint32_t(256 * b + half * HC));
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      if (warp_aborted(abort_flag)) break;
      // rows beyond M and columns beyond N hold padding (scales of padding rows
      // are not written: only live ones may be used)
      const int ea = m < P.M ? P.ea[m] : 0;
      const bool part = P.splits > 1, scale = P.alpha != 1.0;
      const int64_t sm = part ? P.N : P.cm, sn = part ? 1 : P.cn;
      const int64_t mrow = T.m0 + quarter * 32;
      const int rows = int(min(int64_t(32), P.M - mrow));
#pragma unroll
      for (int b = 0; b < Cfg::pair; ++b) {
        const int64_t nb = T.n0 + b * BN + half * HC;
        const int live = int(min(int64_t(HC), P.N - nb));
        if (live <= 0) continue;
        const int* ebp = P.eb + nb;
        auto eb = [&](int j) { return j < live ? __ldg(ebp + j) : 0; };
        double* out = (part ? P.work + int64_t(T.z) * P.M * P.N : P.C) + mrow * sm + nb * sn;
        double v[HC];
        sums[b].values(ea, eb, T.nk * kBK, v);
        if (scale) {
#pragma unroll
          for (int j = 0; j < HC; ++j) v[j] *= P.alpha;
        }
        if (sn != 1) {  // a lane's neighbours are adjacent in memory
#pragma unroll
          for (int j = 0; j < HC; ++j)
            if (j < live && lane < rows) out[lane * sm + j * sn] = v[j];
        } else {
          // Rows of C: a store per column of a lane's row touches 32 sectors with 8
          // bytes each; through the warp's [32][4] piece of shared memory it
          // writes whole sectors, 4 columns of 8 rows at a time.
          double* buf = reinterpret_cast<double*>(smem + Cfg::xpose) + (warp - 1 - Cfg::issuers) * 128;
          const int r0 = lane >> 2, c = lane & 3;
#pragma unroll
          for (int j0 = 0; j0 < HC; j0 += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) buf[lane * 4 + ((u + (lane >> 2)) & 3)] = v[j0 + u];
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int r = u * 8 + r0;
              const double x = buf[r * 4 + ((c + (r >> 2)) & 3)];
              if (r < rows && j0 + c < live) out[r * sm + j0 + c] = x;
            }
            __syncwarp();
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::tcols));
  }
}

// ---------------------------------------------------------------- speculative columns
//
// All columns of a selection block in one launch: for every level l and every
// candidate t, member j of its set,
//   C_l[j][t] = w_l aL (aL + 2 aN) - F,
// aL, aN the products of the basis rows (own functions, coarser ones) and F that
// of the factor rows, each an exact 8-digit product.  A tile (128 candidates x
// 48 members of a level) runs its three k ranges through one ring of stages; the
// epilogue turns a range's integer sums into FP64, keeps the partial result in
// shared memory and writes the finished column once.  Separate products were
// ten launches a block (three per level and the combination), each too short to
// fill the chip on a small cell (18 us of fill and epilogue), and moved every
// result through memory four more times: columns of a block on one cell 290 ->
// 163 us, on 2x2x2 2.01 -> 1.76 ms (99 us and 1.57 ms with integer sums and two
// issuing warps), and one launch instead of up to 21 for the digits of the set's
// rows.
// Bound: the tensor cores (0.7 of their measured rate on 2x2x2, the padding of the
// N tiles counted) and the candidates' digit stream (16 bytes a value) from HBM
// (0.76 of the copy rate); persistent CTAs,
// one per SM, the levels in order (the longest k ranges first).
struct OzColSeg {
  const __nv_bfloat16 *A, *B;
  const int *ea, *eb;
  int64_t akst, bkst;
  int nkt;
};
struct OzColLevel {
  OzColSeg seg[3];
  int64_t M, ntm;
  double* C;
  double w;
};
struct OzColParams {
  OzColLevel l[ISDF_MAX_LEVELS];
  int nlev;
  const int* scount;  // members per level
  int* err;
  unsigned long long wait_ns;
};

struct OzColCfg : OzCfg<8, 48> {
  static constexpr int S = 8, BN = 48;
  static constexpr int stash = kBM * BN * 8;  // partial results, FP64
  static constexpr int ring = nst * stage;
  static constexpr int smem = ring + stash + 1024 + 256;  // + barriers, alignment slack
  static_assert(smem <= 232448, "shared memory per CTA");
};

__global__ void __launch_bounds__(OzColCfg::threads, 1) k_oz_columns(const __grid_constant__ OzColParams P) {
  using Cfg = OzColCfg;
  constexpr int S = Cfg::S, BN = Cfg::BN;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  double* stash = reinterpret_cast<double*>(smem + Cfg::ring);  // [BN][128]
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Cfg::ring + Cfg::stash);
  uint64_t* empty = full + Cfg::nst;
  uint64_t* acc_full = empty + Cfg::nst;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* drain = acc_empty + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + Cfg::issuers);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0);  // uniform to the compiler
  const int lane = threadIdx.x % 32;
  if (__syncthreads_or(threadIdx.x == 0 ? *(volatile const int*)P.err : 0)) return;

  // tiles of level l: [t0[l], t0[l + 1]), N tiles fastest
  int64_t t0[ISDF_MAX_LEVELS + 1] = {0};
  int NT[ISDF_MAX_LEVELS], members[ISDF_MAX_LEVELS];
#pragma unroll
  for (int l = 0; l < ISDF_MAX_LEVELS; ++l) {
    members[l] = l < P.nlev ? P.scount[l] : 0;
    NT[l] = (members[l] + BN - 1) / BN;
    t0[l + 1] = t0[l] + (l < P.nlev ? P.l[l].ntm * NT[l] : 0);
  }
  const int64_t ntiles = t0[ISDF_MAX_LEVELS];
  struct Tile {
    int l, nt, members;
    int64_t mt;
  };
  auto tile_at = [&](int64_t t) {
    Tile T{0, 0, 0, 0};
#pragma unroll
    for (int l = 0; l < ISDF_MAX_LEVELS; ++l)
      if (t >= t0[l] && t < t0[l + 1]) {
        T.l = l;
        T.members = members[l];
        T.mt = (t - t0[l]) / NT[l];
        T.nt = int((t - t0[l]) - T.mt * NT[l]);
      }
    return T;
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < Cfg::nst; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], Cfg::issuers);
    }
    mbar_init(acc_full, Cfg::issuers);
    mbar_init(acc_empty, Cfg::epi);
    for (int i = 0; i < Cfg::issuers; ++i) mbar_init(&drain[i], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(Cfg::tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    // ------------------------------------------------ producer
    if (lane == 0) {
      int64_t g = 0;  // stages issued so far (all tiles)
      for (int64_t t = blockIdx.x; t < ntiles && !*(volatile int*)abort_flag; t += gridDim.x) {
        const Tile T = tile_at(t);
        for (int sg = 0; sg < 3 && !*(volatile int*)abort_flag; ++sg) {
          const OzColSeg& Q = P.l[T.l].seg[sg];
          const unsigned char* gA = reinterpret_cast<const unsigned char*>(Q.A) + T.mt * Q.akst * int64_t(Cfg::stageA);
          const unsigned char* gB = reinterpret_cast<const unsigned char*>(Q.B) + T.nt * Q.bkst * int64_t(Cfg::stageB);
          for (int kt = 0; kt < Q.nkt; ++kt, ++g) {
            const int st = int(g % Cfg::nst);
            const int64_t round = g / Cfg::nst;
            if (round > 0 && !mbar_wait(&empty[st], uint32_t((round - 1) & 1), P.err, P.wait_ns)) {
              set_err(P.err, 11);
              *(volatile int*)abort_flag = 1;
              break;
            }
            if (*(volatile int*)abort_flag) break;
            unsigned char* sA = smem + st * Cfg::stage;
            mbar_expect_tx(&full[st], Cfg::stageA + Cfg::stageB);
            bulk_g2s(sA, gA + kt * int64_t(Cfg::stageA), Cfg::stageA, &full[st]);
            bulk_g2s(sA + Cfg::stageA, gB + kt * int64_t(Cfg::stageB), Cfg::stageB, &full[st]);
          }
        }
      }
      if (*(volatile int*)abort_flag) {  // copies issued but never consumed must land before exit
        const int64_t first = g > Cfg::nst ? g - Cfg::nst : 0;
        for (int64_t it = first; it < g; ++it) mbar_wait(&full[it % Cfg::nst], uint32_t((it / Cfg::nst) & 1), nullptr);
      }
    }
  } else if (warp <= Cfg::issuers) {
    // ------------------------------------------------ MMA issuers
    const uint32_t el = elect_one();
    {
      int64_t g = 0, h = 0;  // stages consumed, accumulator chunks handed over (all tiles)
      bool stop = false;
      for (int64_t t = blockIdx.x; t < ntiles && !stop; t += gridDim.x) {
        const Tile T = tile_at(t);
        for (int sg = 0; sg < 3 && !stop; ++sg) {
          const int nkt = P.l[T.l].seg[sg].nkt;
          for (int kt = 0; kt < nkt; ++kt, ++g) {
            const int st = int(g % Cfg::nst);
            const int cpos = kt % Cfg::kc;
            if (cpos == 0 && h > 0 && !warp_wait(acc_empty, uint32_t((h - 1) & 1), P.err, P.wait_ns)) {
              set_err(P.err, 12);
              stop = true;
            } else if (!warp_wait(&full[st], uint32_t((g / Cfg::nst) & 1), P.err, P.wait_ns)) {
              set_err(P.err, 13);
              stop = true;
            }
            if (stop) *(volatile int*)abort_flag = 1;
            if (stop || warp_aborted(abort_flag)) {
              stop = true;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t sA = smem_u32(smem + st * Cfg::stage);
            mma_stage<S, BN>(warp - 1, el, tmem, sA, sA + Cfg::stageA, cpos == 0, 1);
            umma_commit(el, &empty[st]);
            if (cpos == Cfg::kc - 1 || kt == nkt - 1) {
              umma_commit(el, acc_full);
              ++h;
            }
          }
        }
      }
      umma_commit(el, &drain[warp - 1]);  // all MMAs issued by this thread complete before tensor memory is freed
      mbar_wait(&drain[warp - 1], 0, nullptr);
    }
  } else {
    // ------------------------------------------------ epilogue warps
    constexpr int HC = BN / (Cfg::epi / 4);  // columns per thread
    const int quarter = warp % 4;            // a warp reads tensor-memory lanes 32 (warp % 4) ..
    const int part = (warp - 1 - Cfg::issuers) / 4;  // which share of the columns
    const int row = quarter * 32 + lane;
    const uint32_t tbase = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(part * HC);
    double* mine = stash + part * HC * kBM + row;
    int64_t h = 0;  // accumulator chunks taken over (all tiles)
    for (int64_t t = blockIdx.x; t < ntiles && !warp_aborted(abort_flag); t += gridDim.x) {
      const Tile T = tile_at(t);
      const OzColLevel& L = P.l[T.l];
      const int64_t m = T.mt * kBM + row;
      const int n0 = T.nt * BN + part * HC;
      const bool live = m < L.M;
      const int last = L.seg[2].nkt ? 2 : L.seg[1].nkt ? 1 : 0;
      for (int sg = 0; sg <= last; ++sg) {
        const OzColSeg& Q = L.seg[sg];
        const int nchunks = (Q.nkt + Cfg::kc - 1) / Cfg::kc;
        if (nchunks == 0 && sg > 0 && sg < last) {  // no coarser functions: the M term is ready
          for (int j = 0; j < HC; ++j) {
            const double a = mine[j * kBM];
            mine[j * kBM] = L.w * (a * a);
          }
          continue;
        }
        OzSums<S, HC> sums;
        sums.clear();
        for (int c = 0; c < nchunks; ++c) {
          if (!warp_wait(acc_full, uint32_t(h & 1), P.err, P.wait_ns)) {
            set_err(P.err, 14);
            *(volatile int*)abort_flag = 1;
            break;
          }
          ++h;
          asm volatile("tcgen05.fence::after_thread_sync;");
          sums.template drain<BN>(tbase);
          asm volatile("tcgen05.fence::before_thread_sync;");
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty);
        }
        if (warp_aborted(abort_flag)) break;
        const int ea = live && nchunks ? Q.ea[m] : 0;
        const int* ebp = Q.eb + n0;
        const int cols = nchunks ? T.members - n0 : 0;  // live ones among this thread's (the others' scales are unset)
        auto eb = [&](int j) { return j < cols ? __ldg(ebp + j) : 0; };
        double v[HC];
        sums.values(ea, eb, int64_t(Q.nkt) * kBK, v);
        if (sg == 1) {
#pragma unroll
          for (int j = 0; j < HC; ++j) {
            const double a = mine[j * kBM];
            v[j] = L.w * (a * (a + 2.0 * v[j]));
          }
        } else if (sg == 2) {
#pragma unroll
          for (int j = 0; j < HC; ++j) v[j] = mine[j * kBM] - v[j];
        } else if (last == 0) {
#pragma unroll
          for (int j = 0; j < HC; ++j) v[j] = L.w * (v[j] * v[j]);
        }
        if (sg < last) {
#pragma unroll
          for (int j = 0; j < HC; ++j) mine[j * kBM] = v[j];
        } else {
          double* out = L.C + int64_t(n0) * L.M + m;
#pragma unroll
          for (int j = 0; j < HC; ++j)
            if (n0 + j < T.members && live) out[int64_t(j) * L.M] = v[j];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::tcols));
  }
}

// Digits of the set's rows on the B side of the three products, all levels: one
// block per member and product.  Basis rows take the scale of the same
// candidate's row on the A side; factor rows their own maximum.
struct OzRowsLevel {
  const double* src[3];  // element (row, k) at src[row + k * ld]
  int64_t ld[3];
  int K[3];
  const int* aexp[2];
  int* bexp[3];
  __nv_bfloat16* tiles[3];
  int64_t kst[3];
};
struct OzRowsParams {
  OzRowsLevel l[ISDF_MAX_LEVELS];
  const int *scount, *st, *sg;  // members per level; candidate and grid point of each
};
__global__ void __launch_bounds__(256) k_oz_set_rows(const __grid_constant__ OzRowsParams P) {
  constexpr int S = 8, BN = 48;
  __shared__ unsigned long long key;
  int j = int(blockIdx.x), l = 0, first = 0;
  const int sg = int(blockIdx.y), tid = threadIdx.x;
  while (l < ISDF_MAX_LEVELS && j >= first + P.scount[l]) first += P.scount[l], ++l;
  if (l == ISDF_MAX_LEVELS) return;  // fewer members than the set's size
  const OzRowsLevel& L = P.l[l];
  const int K = L.K[sg], r = j - first;
  const int ngrp = ((K + kBK - 1) / kBK) * (kBK / 8);
  if (!K) return;
  const int64_t ld = L.ld[sg];
  const double* row = L.src[sg] + (sg == 2 ? P.st[j] : P.sg[j]);
  double v[8];
  int e;
  if (sg < 2) {
    e = L.aexp[sg][P.st[j]];
  } else {
    if (tid == 0) key = 0ull;
    __syncthreads();
    uint64_t m = 0;
    for (int g = tid; g < ngrp; g += 256) {
      oz_load8(row, true, ld, K, g, v);
#pragma unroll
      for (int u = 0; u < 8; ++u) m = umax64(m, abs_key(v[u]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = umax64(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0 && m) atomicMax(&key, (unsigned long long)m);
    __syncthreads();
    e = exp_of_key(key);
  }
  if (tid == 0) L.bexp[sg][r] = e;
  for (int g = tid; g < ngrp; g += 256) {
    if (sg < 2 || ngrp > 256) oz_load8(row, true, ld, K, g, v);
    __nv_bfloat16* out = L.tiles[sg] + ((r / BN * L.kst[sg] + g / (kBK / 8)) * S) * int64_t(BN * kBK) +
                         oz_inner(r % BN, g % (kBK / 8));
    oz_digits8<S>(v, 7 * S - e, BN * kBK, out);
  }
}

// C = sum_z work[z] (deterministic order), same store maps as the GEMM
__global__ void k_oz_reduce(const double* __restrict__ work, int splits, int64_t M, int64_t N, double* __restrict__ C,
                            int64_t cm, int64_t cn, int sym) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= M * N) return;
  const int64_t m = e / N, n = e % N;
  if (sym && n > m) return;
  double s = 0.0;
  for (int z = 0; z < splits; ++z) s += work[int64_t(z) * M * N + e];
  C[m * cm + n * cn] = s;
}

// persistent: one wave of CTAs that loop over the tiles (a tile's epilogue
// then overlaps the next tile's copies and MMAs); else one CTA per tile, the
// hardware scheduler balancing tiles of uneven length (split or triangular
// products) across the SMs.
template <int S, int BN>
void launch_oz(const OzGemmParams& P, bool persistent, cudaStream_t s) {
  using Cfg = OzCfg<S, BN>;
  // the shared-memory attributes belong to the current device: set them, and
  // count the CTAs of this configuration the device holds at once, per device
  static std::atomic<int> resident[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    dev = 0;
  }
  int res = resident[dev].load(std::memory_order_acquire);
  if (!res) {
    cudaFuncSetAttribute(k_oz_gemm<S, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::smem);
    cudaFuncSetAttribute(k_oz_gemm<S, BN>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    int nsm = 0, per = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_oz_gemm<S, BN>, Cfg::threads, Cfg::smem);
    cudaGetLastError();
    res = std::max(1, nsm) * std::max(1, per);
    resident[dev].store(res, std::memory_order_release);
  }
  const int64_t ntiles = ((P.ntn + Cfg::pair - 1) / Cfg::pair) * P.ntm * P.splits;
  const unsigned grid = unsigned(std::max<int64_t>(1, persistent ? std::min<int64_t>(ntiles, res) : ntiles));
  k_oz_gemm<S, BN><<<grid, Cfg::threads, Cfg::smem, s>>>(P);
}

}  // namespace

int64_t oz_tile_bytes(const OzOperand& op) { return op.nrt * op.kst * op.S * int64_t(op.rt) * kBK * 2; }

int64_t oz_tile_elems(int64_t rows, int64_t K, int rt, int S) {
  const int64_t nrt = (rows + rt - 1) / rt, nkt = (K + kBK - 1) / kBK;
  return nrt * nkt * S * int64_t(rt) * kBK;
}

isdf_status oz_alloc(Plan* p, OzOperand& op, int64_t rows, int64_t K, int rt, int S, const char* what) {
  op.rows = rows;
  op.K = K;
  op.tiles = nullptr;
  op.exps = nullptr;
  op.rt = rt;
  op.S = S;
  op.nrt = (rows + rt - 1) / rt;
  op.nkt = (K + kBK - 1) / kBK;
  op.kst = op.nkt;
  isdf_status st = dalloc(p, &op.tiles, size_t(oz_tile_elems(rows, K, rt, S)) * 2, what);
  if (st) return st;
  return dalloc_t(p, &op.exps, size_t(op.nrt * rt), what);
}

void oz_free(OzOperand& op) {
  dfree(op.tiles);
  dfree(op.exps);
  op.tiles = nullptr;
  op.exps = nullptr;
}

void oz_slice(const double* src, int64_t sr, int64_t sk, const double* kw, double mul, OzOperand& op, cudaStream_t s) {
  slice_operand(slice_args(src, sr, sk, kw, mul, nullptr, op, 0, op.nkt * (kBK / 8)), op.S, s);
}

unsigned long long* oz_keys_begin(OzOperand& op, cudaStream_t s) {
  cudaMemsetAsync(op.tiles, 0, sizeof(unsigned long long) * size_t(op.rows), s);
  return static_cast<unsigned long long*>(op.tiles);
}

void oz_slice_keyed(const double* src, int64_t sr, OzOperand& op, cudaStream_t s) {
  const OzSliceArgs A = slice_args(src, sr, 1, nullptr, 1.0, nullptr, op, 0, op.nkt * (kBK / 8));
  k_oz_key_exps<<<unsigned((op.rows + 255) / 256), 256, 0, s>>>(static_cast<unsigned long long*>(op.tiles), op.rows,
                                                                op.exps);
  count_launches(1);
  launch_digits(A, op.S, s);
}

void oz_slice_ex(const double* src, int64_t sr, int64_t sk, const int* ridx, OzOperand& op, int64_t kg0, int64_t kg1,
                 bool exps_ready, cudaStream_t s) {
  if (op.rows <= 0 || kg1 <= kg0) return;
  const OzSliceArgs A = slice_args(src, sr, sk, nullptr, 1.0, ridx, op, kg0, kg1 - kg0);
  if (exps_ready)
    launch_digits(A, op.S, s);
  else
    slice_operand(A, op.S, s);  // scales need every group: callers pass the whole range
}

// host-side fault injection (ISDF_FAULT=oz_wait): every pipeline wait gives
// up at once, so the launch takes its error path (error code, copies and
// MMAs in flight completed, tensor memory freed) and the call reports
// ISDF_ERR_TIMEOUT; nothing faults or hangs
static unsigned long long oz_wait_limit() {
  const char* fault = std::getenv("ISDF_FAULT");
  return (fault && std::strcmp(fault, "oz_wait") == 0) ? 0ull : kWaitNs;
}

int oz_bn(int S) { return oz_tile_n(S); }

void oz_gemm(const OzOperand& A, const OzOperand& B, double* C, int64_t ldc, int trans, double alpha, int tri, int sym,
             int splits, double* work, int* err, cudaStream_t s, const OzWindows* win) {
  OzGemmParams P;
  if (win) P.win = *win;
  P.A = static_cast<const __nv_bfloat16*>(A.tiles);
  P.B = static_cast<const __nv_bfloat16*>(B.tiles);
  P.ea = A.exps;
  P.eb = B.exps;
  P.M = A.rows;
  P.N = B.rows;
  P.nkt = A.nkt;
  P.akst = A.kst > 0 ? A.kst : A.nkt;
  P.bkst = B.kst > 0 ? B.kst : B.nkt;
  P.bgroups = B.rt == oz_bn(B.S) ? 0 : B.nrt * (kBM / 8);
  P.tri = tri;
  P.sym = sym;
  P.splits = splits < 1 ? 1 : splits;
  P.C = C;
  P.cm = trans ? 1 : ldc;
  P.cn = trans ? ldc : 1;
  P.alpha = alpha;
  P.work = work;
  P.err = err;
  P.wait_ns = oz_wait_limit();
  P.ntm = A.nrt;
  P.ntn = (B.rows + oz_bn(B.S) - 1) / oz_bn(B.S);
  // Persistent CTAs pay off where a tile's epilogue is long against its main
  // loop (it then runs under the next tile's): with 5 digits, and with the exact
  // epilogues over short K (131072 x 48 x 512, 8 digits: 291 -> 213 us); long,
  // split or triangular exact products are faster with one CTA per tile, balanced
  // by the hardware scheduler.
  const bool persistent = A.S == 5 || (A.S >= 7 && P.splits == 1 && !P.sym && P.tri == 0 && P.nkt * kBK <= 4096);
  if (A.S == 5)
    launch_oz<5, 48>(P, persistent, s);
  else if (A.S == 8)
    launch_oz<8, 48>(P, persistent, s);
  else if (A.S == 7)
    launch_oz<7, 48>(P, persistent, s);
  else
    launch_oz<6, 64>(P, persistent, s);
  count_launches(1);
  if (P.splits > 1) {
    const int64_t tot = A.rows * B.rows;
    k_oz_reduce<<<unsigned((tot + 255) / 256), 256, 0, s>>>(work, P.splits, A.rows, B.rows, C, P.cm, P.cn, sym);
    count_launches(1);
  }
}

void oz_set_rows(const OzColumnJob* jobs, int nlev, int smax, const int* scount, const int* st, const int* sg,
                 cudaStream_t s) {
  OzRowsParams P{};
  P.scount = scount;
  P.st = st;
  P.sg = sg;
  bool factor = false;
  for (int l = 0; l < nlev; ++l) {
    const OzColumnJob& J = jobs[l];
    OzRowsLevel& L = P.l[l];
    for (int q = 0; q < 3; ++q) {
      if (!J.A[q] || J.A[q]->nkt == 0 || J.A[q]->rows == 0) continue;
      L.src[q] = J.src[q];
      L.ld[q] = J.ld[q];
      L.K[q] = int(J.A[q]->K);
      if (q < 2) L.aexp[q] = J.A[q]->exps;
      L.bexp[q] = J.B[q]->exps;
      L.tiles[q] = static_cast<__nv_bfloat16*>(J.B[q]->tiles);
      L.kst[q] = J.B[q]->kst;
      factor = factor || q == 2;
    }
  }
  k_oz_set_rows<<<dim3(unsigned(smax), factor ? 3u : 2u), 256, 0, s>>>(P);
  count_launches(1);
}

void oz_columns(const OzColumnJob* jobs, int nlev, const int* scount, int* err, cudaStream_t s) {
  static std::atomic<int> sms[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    dev = 0;
  }
  int n = sms[dev].load(std::memory_order_acquire);
  if (!n) {
    cudaFuncSetAttribute(k_oz_columns, cudaFuncAttributeMaxDynamicSharedMemorySize, OzColCfg::smem);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    n = std::max(1, n);
    sms[dev].store(n, std::memory_order_release);
  }
  OzColParams P{};
  P.nlev = nlev;
  P.scount = scount;
  P.err = err;
  P.wait_ns = oz_wait_limit();
  for (int l = 0; l < nlev; ++l) {
    const OzColumnJob& J = jobs[l];
    OzColLevel& L = P.l[l];
    L.M = J.M;
    L.ntm = (J.M + kBM - 1) / kBM;
    L.C = J.C;
    L.w = J.w;
    for (int q = 0; q < 3; ++q) {
      if (!J.A[q] || J.A[q]->nkt == 0) continue;
      L.seg[q] = {static_cast<const __nv_bfloat16*>(J.A[q]->tiles), static_cast<const __nv_bfloat16*>(J.B[q]->tiles),
                  J.A[q]->exps, J.B[q]->exps, J.A[q]->kst, J.B[q]->kst, int(J.A[q]->nkt)};
    }
  }
  k_oz_columns<<<unsigned(n), OzColCfg::threads, OzColCfg::smem, s>>>(P);
  count_launches(1);
}

// ---------------------------------------------------------------- split-K autotuner
//
// The one free launch parameter of a product shape is its split-K factor
// (how many CTAs share one output tile's k range).  On the first product of
// a shape (rows of A, rows of B, k tiles, digits, symmetric or not) outside
// any graph capture (products of more than 0.3 ms follow oz_rule_splits
// instead), every admissible candidate runs on the real operands
// (one warm-up run, then one timed run per candidate, CUDA events on the
// product's stream) and the fastest is cached for the process; the heuristic's choice
// is among the candidates, and the chosen one runs last so C holds its
// result.  Candidates whose split-K partials would exceed 2 GiB are skipped.

namespace {
struct TuneKey {
  int64_t M, N, nkt;
  int S, sym, trans;
  bool operator<(const TuneKey& o) const {
    return std::tie(M, N, nkt, S, sym, trans) < std::tie(o.M, o.N, o.nkt, o.S, o.sym, o.trans);
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, std::pair<int, float>> g_tune;  // shape -> (splits, ms)
}  // namespace

int oz_tuned_splits(Plan* p, const OzOperand& A, const OzOperand& B, double* C, int64_t ldc, int trans, int sym,
                    int heuristic, cudaStream_t s, const OzWindows* win) {
  const TuneKey key{A.rows, B.rows, A.nkt, A.S, sym | (win ? 2 << win->side : 0), trans};
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) return it->second.first;
  }
  if ((p && p->capturing) || std::getenv("ISDF_NO_AUTOTUNE")) return heuristic;
  if (!win)
    if (const int c = oz_rule_splits(A.rows, B.rows, A.nkt, A.S, sym != 0)) return c;
  std::vector<int> cand;
  for (int c : {1, 2, 4, 8, 16, 32, 64})
    if (c <= std::max<int64_t>(1, A.nkt)) cand.push_back(c);
  if (std::find(cand.begin(), cand.end(), heuristic) == cand.end()) cand.push_back(heuristic);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  int* err = p ? p->d_ozerr : nullptr;
  int best = heuristic;
  float best_ms = 1e30f;
  for (int c : cand) {
    double* work = nullptr;
    if (!oz_splits_fit(c, A.rows, B.rows)) continue;
    const size_t wbytes = c > 1 ? sizeof(double) * size_t(c) * A.rows * B.rows : 0;
    if (wbytes && cudaMallocAsync(reinterpret_cast<void**>(&work), wbytes, s) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    float ms = 1e30f;
    for (int rep = (c == cand.front() ? 0 : 1); rep < 2; ++rep) {  // one warm-up run before the first candidate
      cudaEventRecord(e0, s);
      oz_gemm(A, B, C, ldc, trans, 1.0, 0, sym, c, work, err, s, win);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float t = 0.0f;
      if (rep > 0 && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms = std::min(ms, t);
    }
    if (work) cudaFreeAsync(work, s);
    if (ms < best_ms) best_ms = ms, best = c;
  }
  int herr = 0;  // after an expired wait the products return at once: no times to keep
  if (err) cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaGetLastError();
  if (herr) return heuristic;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune[key] = {best, best_ms};
  return best;
}

std::string oz_tune_json() {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  std::string o = "[";
  for (const auto& kv : g_tune) {
    if (o.size() > 1) o += ",";
    o += "{\"M\":" + std::to_string(kv.first.M) + ",\"N\":" + std::to_string(kv.first.N) +
         ",\"k_tiles\":" + std::to_string(kv.first.nkt) + ",\"digits\":" + std::to_string(kv.first.S) +
         ",\"sym\":" + std::to_string(kv.first.sym & 1) + ",\"splits\":" + std::to_string(kv.second.first) +
         ",\"ms\":" + std::to_string(kv.second.second) + "}";
  }
  return o + "]";
}

// ------------------------------------------------------- stand-alone products
//
// gemm_alloc takes its scratch from the pool of the calls without a plan;
// gemm_noalloc runs the same kernels on one file-scope device array, which
// every GPU that loads the library holds until the process exits.

constexpr size_t kStaticScratchBytes = size_t(32) << 20;
static __device__ __align__(256) unsigned char g_gemm_static_scratch[kStaticScratchBytes];

namespace {

std::mutex g_static_mu;
void* g_static_addr[kMaxDevices] = {nullptr};

size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// Where a stand-alone product keeps its operands in one block of scratch.
struct GemmScratch {
  OzOperand a, b;
  size_t a_exps, b_tiles, b_exps, err, work, bytes;
  GemmScratch(int64_t M, int64_t N, int64_t K, int slices, int splits) {
    a.rows = M, a.rt = 128, b.rows = N, b.rt = oz_bn(slices);
    for (OzOperand* o : {&a, &b})
      o->K = K, o->S = slices, o->nrt = (o->rows + o->rt - 1) / o->rt, o->nkt = o->kst = (K + kBK - 1) / kBK;
    a_exps = round256(size_t(oz_tile_elems(M, K, a.rt, slices)) * 2);
    b_tiles = a_exps + round256(sizeof(int) * size_t(a.nrt * a.rt));
    b_exps = b_tiles + round256(size_t(oz_tile_elems(N, K, b.rt, slices)) * 2);
    err = b_exps + round256(sizeof(int) * size_t(b.nrt * b.rt));
    work = err + 256;
    bytes = work + (splits > 1 ? sizeof(double) * size_t(splits) * M * N : 0);
  }
  // the arrays from base on; the error word is to be cleared by the caller
  void place(unsigned char* base) {
    a.tiles = base, a.exps = reinterpret_cast<int*>(base + a_exps);
    b.tiles = base + b_tiles, b.exps = reinterpret_cast<int*>(base + b_exps);
  }
};

// The product on scratch at base; `name` is the entry point, for messages.
isdf_status gemm_on(GemmScratch& g, unsigned char* base, const double* A, const double* B, double* C, int64_t lda,
                    int64_t ldb, int64_t ldc, double alpha, int splits, cudaStream_t s, const char* name,
                    std::string& why) {
  g.place(base);
  int* err = reinterpret_cast<int*>(base + g.err);
  // the block keeps an earlier call's contents: the error word must start at
  // zero; every slice byte and every scale read below is rewritten first.
  // Clear any stale launch error so the check after the launches sees ours.
  cudaGetLastError();
  if (cudaMemsetAsync(err, 0, sizeof(int), s) != cudaSuccess) {
    cudaGetLastError();
    why = std::string(name) + ": cudaMemsetAsync of the error word failed";
    return ISDF_ERR_CUDA;
  }
  oz_slice(A, lda, 1, nullptr, 1.0, g.a, s);
  oz_slice(B, ldb, 1, nullptr, 1.0, g.b, s);
  oz_gemm(g.a, g.b, C, ldc, 0, alpha, 0, 0, splits, splits > 1 ? reinterpret_cast<double*>(base + g.work) : nullptr, err,
          s);
  // a launch that could not start (configuration, resources) is reported here
  // and nowhere else: the copy below would succeed with C unwritten
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    why = std::string(name) + ": launch failed: " + cudaGetErrorString(e);
    return ISDF_ERR_CUDA;
  }
  int herr = 0;
  e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    why = std::string(name) + ": " + cudaGetErrorString(e);
    return ISDF_ERR_CUDA;
  }
  if (herr) {
    why = std::string(name) + ": tensor-core pipeline wait expired (code " + std::to_string(herr) + ")";
    return ISDF_ERR_TIMEOUT;
  }
  return ISDF_OK;
}

}  // namespace

isdf_status gemm_alloc(const double* A, const double* B, double* C, int64_t M, int64_t N, int64_t K, int64_t lda,
                       int64_t ldb, int64_t ldc, double alpha, int slices, int splits, cudaStream_t s,
                       std::string& why) {
  GemmScratch g(M, N, K, slices, splits);
  void* base = nullptr;
  const cudaError_t e = scratch_alloc(&base, g.bytes, s);
  if (e != cudaSuccess) {
    why = std::string("isdf_gemm_f64: allocation failed: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? ISDF_ERR_OOM : ISDF_ERR_CUDA;
  }
  const isdf_status st = gemm_on(g, static_cast<unsigned char*>(base), A, B, C, lda, ldb, ldc, alpha, splits, s,
                                 "isdf_gemm_f64", why);
  scratch_free(base, s);
  return st;
}

size_t gemm_noalloc_capacity() { return kStaticScratchBytes; }

isdf_status gemm_noalloc(const double* A, const double* B, double* C, int64_t M, int64_t N, int64_t K, int64_t lda,
                         int64_t ldb, int64_t ldc, double alpha, int slices, cudaStream_t s, std::string& why) {
  // bound every extent by the array before any size arithmetic: with each of
  // M, N, K at most the array's byte count the products below cannot overflow
  const int64_t cap = int64_t(kStaticScratchBytes);
  if (M > cap || N > cap || K > cap || M * K > cap || N * K > cap) {
    why = "isdf_gemm_f64_noalloc: operands of " + std::to_string(M) + " x " + std::to_string(K) + " and " +
          std::to_string(N) + " x " + std::to_string(K) + " exceed what the static array holds (" +
          std::to_string(kStaticScratchBytes) + " bytes)";
    return ISDF_ERR_ARG;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    why = "no current CUDA device";
    return ISDF_ERR_CUDA;
  }
  unsigned char* base = nullptr;
  {
    // set-up once per device, with that device current: the array's name is
    // a host-side stand-in, its device address comes from the runtime
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_addr[dev]) {
      void* ptr = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&ptr, g_gemm_static_scratch);
      if (e != cudaSuccess || !ptr) {
        cudaGetLastError();
        why = std::string("cudaGetSymbolAddress of the static scratch failed: ") + cudaGetErrorString(e);
        return ISDF_ERR_CUDA;
      }
      g_static_addr[dev] = ptr;
    }
    base = static_cast<unsigned char*>(g_static_addr[dev]);
  }
  GemmScratch g(M, N, K, slices, 1);
  if (g.bytes > kStaticScratchBytes) {
    why = "isdf_gemm_f64_noalloc needs " + std::to_string(g.bytes) + " bytes of scratch; the static array holds " +
          std::to_string(kStaticScratchBytes);
    return ISDF_ERR_ARG;
  }
  return gemm_on(g, base, A, B, C, lda, ldb, ldc, alpha, 1, s, "isdf_gemm_f64_noalloc", why);
}

}  // namespace isdf
