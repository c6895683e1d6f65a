// Interpolation-point selection (kernel family (b)): greedy pivoted Cholesky on
// the block-diagonal matrix (+)_l w_l M_l (Section II.A, Eq. 2).
//
// The loop stays on the device: each step is two kernels that read and write
// a small state record, so the pivot index never travels to the host.
//   k_sel_first  stop rules; tie rule: smallest global index with d >= thr
//                (atomicMin); the last block to contribute records the pivot,
//                advances counters and checks the device-clock time budget
//   k_sel_col    new factor column on the pivot's level and residual update:
//                L[g,k] = (w M(g,p) - sum_j L[g,j] L[p,j]) / sqrt(d_p),
//                d(g) -= L[g,k]^2,  L[p,k] = sqrt(d_p), d(p) = 0;
//                and the level's largest residual (atomicMax on the bit
//                pattern, d >= 0), which k_sel_max finds before the first step
// Steps are captured once into a CUDA graph and replayed.  No kernel waits on
// another; there is no spin anywhere.
//
// Candidates.  Every level works on a compacted, ascending list of candidate
// grid points (all points, a caller-given list, or the exact prefilter), so
// the factor columns, the residual and every step scale with the number of
// candidates.  Exact prefilter: a point whose initial residual is below tau
// can never be picked while every pivot value stays above tau plus the tie
// margin, because residuals only shrink; the host checks that certificate on
// the returned pivot values and otherwise repeats with a lower tau.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

#include "dfloat.cuh"
#include "digits.cuh"
#include "internal.cuh"

namespace isdf {
namespace {

struct SelState {
  unsigned long long lmax[ISDF_MAX_LEVELS];  // largest residual of every level (bits; >= 0)
  unsigned long long first;
  unsigned int arrived;  // blocks of k_sel_first that have contributed
  double d0;
  double dp;
  long long gp;  // grid index of this step's pivot
  long long tp;  // its position in the level's candidate list
  int lev;
  int col;
  int k;
  int done;  // no further steps
  int skip;  // this step has no pivot
  int err;
  int kl[ISDF_MAX_LEVELS];
  unsigned long long t0;
  // speculative blocks
  int final_;                // a stop rule ended the selection
  int bsteps;                // steps accepted in the current round of a block
  int members[ISDF_MAX_LEVELS];  // the block's set, per level
};

struct SelParams {
  double* d;  // residual over all levels' candidates (concatenated)
  int64_t ntot;
  int nlev;
  int64_t coff[ISDF_MAX_LEVELS + 1];  // candidate offsets per level
  const int* cidx[ISDF_MAX_LEVELS];   // candidate grid indices (nullptr: all points)
  int64_t nc[ISDF_MAX_LEVELS];
  double* fac[ISDF_MAX_LEVELS];       // factor columns [col][nc]
  const double* phi[ISDF_MAX_LEVELS];
  int64_t ng[ISDF_MAX_LEVELS];
  int nL[ISDF_MAX_LEVELS];
  int nG[ISDF_MAX_LEVELS];
  double w[ISDF_MAX_LEVELS];
  int64_t* piv;
  double* dval;
  int nip;
  double tol, tie_rel, tie_abs;
  unsigned long long timeout_ns;
};

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

template <class T, class Op>
__device__ __forceinline__ T block_reduce(T v, Op op, T* sh) {
  for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  if (wid == 0) {
    v = (lane < nw) ? sh[lane] : sh[0];
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

struct MaxOp {
  __device__ double operator()(double a, double b) const { return fmax(a, b); }
};
struct MaxU64 {
  __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a > b ? a : b; }
};
struct MinOp {
  __device__ unsigned long long operator()(unsigned long long a, unsigned long long b) const { return a < b ? a : b; }
};

// w_l M_l(g, g) = w (aL^2 + 2 aL aN), aX = sum_{mu in X} phi_mu(g)^2, every grid point
__global__ void k_sel_diag(const double* __restrict__ phi, int64_t ng, int nL, int nG, double w,
                           double* __restrict__ d) {
  for (int64_t g = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; g < ng; g += int64_t(gridDim.x) * blockDim.x) {
    double aL = 0.0, aN = 0.0;
    for (int r = 0; r < nL; ++r) {
      const double v = phi[int64_t(r) * ng + g];
      aL = fma(v, v, aL);
    }
    for (int r = nL; r < nG; ++r) {
      const double v = phi[int64_t(r) * ng + g];
      aN = fma(v, v, aN);
    }
    d[g] = w * (aL * (aL + 2.0 * aN));
  }
}

// max of a vector into a scalar slot (slot preset to 0; values >= 0 compare as bits)
__global__ void k_vec_max(const double* __restrict__ v, int64_t n, unsigned long long* out) {
  __shared__ double sh[32];
  double m = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    m = fmax(m, v[i]);
  m = block_reduce(m, MaxOp(), sh);
  if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// ordered compaction of {g : d0[g] >= tau}: per-block counts, then scatter
constexpr int kCompactBlock = 1024;
__global__ void k_flag_count(const double* __restrict__ d0, int64_t ng, double tau, int* __restrict__ counts) {
  __shared__ int sh[32];
  const int64_t g = int64_t(blockIdx.x) * kCompactBlock + threadIdx.x;
  const int f = (g < ng && d0[g] >= tau) ? 1 : 0;
  const unsigned b = __ballot_sync(0xffffffffu, f);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = __popc(b);
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    for (int i = 0; i < kCompactBlock / 32; ++i) c += sh[i];
    counts[blockIdx.x] = c;
  }
}

__global__ void k_compact(const double* __restrict__ d0, int64_t ng, double tau, const int* __restrict__ block_off,
                          int* __restrict__ cidx) {
  __shared__ int warp_off[32];
  const int64_t g = int64_t(blockIdx.x) * kCompactBlock + threadIdx.x;
  const int f = (g < ng && d0[g] >= tau) ? 1 : 0;
  const unsigned b = __ballot_sync(0xffffffffu, f);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) warp_off[wid] = __popc(b);
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int i = 0; i < kCompactBlock / 32; ++i) {
      const int c = warp_off[i];
      warp_off[i] = acc;
      acc += c;
    }
  }
  __syncthreads();
  if (f) cidx[block_off[blockIdx.x] + warp_off[wid] + __popc(b & ((1u << lane) - 1u))] = int(g);
}

// residual over the candidates of one level
__global__ void k_gather_diag(const double* __restrict__ d0, const int* __restrict__ cidx, int64_t nc,
                              double* __restrict__ d) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < nc) d[t] = d0[cidx ? cidx[t] : t];
}

// Largest residual of every level, before the first step; from then on k_sel_col
// keeps its level's.  blockIdx.y: the level.
__global__ void k_sel_max(SelParams P, SelState* st) {
  if (st->done) return;
  __shared__ double sh[32];
  const int l = blockIdx.y;
  double m = 0.0;
  for (int64_t i = P.coff[l] + int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < P.coff[l + 1];
       i += int64_t(gridDim.x) * blockDim.x)
    m = fmax(m, P.d[i]);
  m = block_reduce(m, MaxOp(), sh);
  if (threadIdx.x == 0 && m > 0.0) atomicMax(&st->lmax[l], (unsigned long long)__double_as_longlong(m));
}

__device__ __forceinline__ double sel_dmax(const SelState* st) {
  unsigned long long m = 0ull;
#pragma unroll
  for (int l = 0; l < ISDF_MAX_LEVELS; ++l) m = max(m, st->lmax[l]);
  return __longlong_as_double((long long)m);
}

// The pivot of the step whose smallest qualifying index is known; one thread.
__device__ __forceinline__ void sel_pick(const SelParams& P, SelState* st, unsigned long long idx, double dmax) {
  if (idx == ULLONG_MAX) {  // nothing qualifies: the largest residual is infinite, its tie threshold not a number
    st->done = 1;
    st->skip = 1;
    st->final_ = 1;
    return;
  }
  int l = 0;
  while (l + 1 < P.nlev && (long long)idx >= P.coff[l + 1]) ++l;
  const long long t = (long long)idx - P.coff[l];
  const long long g = P.cidx[l] ? P.cidx[l][t] : t;
  const double dp = P.d[idx];
  const int k = st->k;
  if (k == 0) st->d0 = dmax;
  st->lev = l;
  st->gp = g;
  st->tp = t;
  st->dp = dp;
  st->col = st->kl[l];
  P.piv[k] = ((long long)l << kPivShift) | g;
  P.dval[k] = dp;
  st->kl[l] += 1;
  st->k = k + 1;
  st->skip = 0;
  st->lmax[l] = 0ull;  // k_sel_col puts the level's new one here
  if (P.timeout_ns) {
    const unsigned long long now = globaltimer();
    if (k == 0) {
      st->t0 = now;
    } else if (now - st->t0 > P.timeout_ns) {
      st->err = ISDF_ERR_TIMEOUT;
      st->done = 1;  // this step's column is still computed
    }
  }
}

// Blocks of the passes over all residuals: one value a thread as far as four blocks an SM go
unsigned sel_blocks(int64_t ntot, int nsm) {
  return unsigned(std::max<int64_t>(1, std::min<int64_t>(int64_t(nsm) * 4, (ntot + 255) / 256)));
}

// The step's pivot: smallest index within the tie window of the largest
// residual; the last block to contribute records it.  Launches of a few
// microseconds bound a step of a small cell: with max, first, pick and column as
// four of them, one cell on a 24^3 grid took 13.9 ms for 312 steps and its fit,
// now 10.9 ms.
__global__ void k_sel_first(SelParams P, SelState* st) {
  if (st->done) return;
  __shared__ unsigned long long sh[32];
  const double dmax = sel_dmax(st);
  const int k = st->k;
  const double d0 = (k == 0) ? dmax : st->d0;
  const bool stop = (k >= P.nip) || !(dmax > 0.0) || (dmax < P.tol * d0);
  if (stop) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      st->done = 1;
      st->skip = 1;
      st->final_ = 1;
    }
    return;
  }
  const double thr = dmax - fmax(P.tie_rel * dmax, P.tie_abs * d0);
  unsigned long long best = ULLONG_MAX;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < P.ntot; i += int64_t(gridDim.x) * blockDim.x) {
    const double v = P.d[i];
    if (v >= thr && v > 0.0) {
      best = (unsigned long long)i;
      break;  // grid-stride order: the first hit is this thread's smallest
    }
  }
  best = block_reduce(best, MinOp(), sh);
  if (threadIdx.x != 0) return;
  if (best != ULLONG_MAX) atomicMin(&st->first, best);
  __threadfence();
  if (atomicAdd(&st->arrived, 1u) + 1u < gridDim.x) return;
  // every other block has read the state and left its index
  __threadfence();
  const unsigned long long idx = atomicExch(&st->first, ULLONG_MAX);
  st->arrived = 0u;
  sel_pick(P, st, idx, dmax);
}

// One block works on 32 candidate points at a time (one point per lane, so
// every load is a coalesced row segment); its 8 warps split the basis
// functions and factor columns 8 ways and the partial dot products are added
// in shared memory in a fixed order.  Grid-striding over 32-point groups keeps
// every SM equally busy whatever the number of candidates.
constexpr int kColWarps = 8;
__global__ __launch_bounds__(32 * kColWarps) void k_sel_col(SelParams P, SelState* st) {
  if (st->skip) return;
  extern __shared__ double sm[];
  const int l = st->lev;
  const int nL = P.nL[l], nG = P.nG[l];
  double* cp = sm;                                 // phi_G(p)
  double* part = sm + ((nG + 1) & ~1);             // [3][kColWarps][32]
  const int64_t gp = st->gp, tp = st->tp;
  const int col = st->col;
  const double dp = st->dp;
  const int64_t ng = P.ng[l], nc = P.nc[l];
  const int* __restrict__ cidx = P.cidx[l];
  const double* __restrict__ phi = P.phi[l];
  double* __restrict__ fac = P.fac[l];
  double* __restrict__ d = P.d + P.coff[l];
  for (int r = threadIdx.x; r < nG; r += blockDim.x) cp[r] = phi[int64_t(r) * ng + gp];
  __syncthreads();
  const double sq = sqrt(dp);
  const double w = P.w[l];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ngroups = (nc + 31) / 32;
  double dmax = 0.0;  // of this lane's candidates, warp 0
  for (int64_t grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    const int64_t t = grp * 32 + lane;
    const bool valid = t < nc;
    double aL = 0.0, aN = 0.0, s = 0.0;
    if (valid) {
      const int64_t g = cidx ? cidx[t] : t;
      // independent partial sums keep several loads and FMAs in flight
      double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0;
      int r = warp;
      for (; r + kColWarps < nL; r += 2 * kColWarps) {
        a0 = fma(phi[int64_t(r) * ng + g], cp[r], a0);
        a1 = fma(phi[int64_t(r + kColWarps) * ng + g], cp[r + kColWarps], a1);
      }
      if (r < nL) a0 = fma(phi[int64_t(r) * ng + g], cp[r], a0);
      r = nL + warp;
      for (; r + kColWarps < nG; r += 2 * kColWarps) {
        b0 = fma(phi[int64_t(r) * ng + g], cp[r], b0);
        b1 = fma(phi[int64_t(r + kColWarps) * ng + g], cp[r + kColWarps], b1);
      }
      if (r < nG) b0 = fma(phi[int64_t(r) * ng + g], cp[r], b0);
      aL = a0 + a1;
      aN = b0 + b1;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      const double* fp = fac + tp;
      const double* ft = fac + t;
      int j = warp;
      for (; j + 3 * kColWarps < col; j += 4 * kColWarps) {
        s0 = fma(ft[int64_t(j) * nc], fp[int64_t(j) * nc], s0);
        s1 = fma(ft[int64_t(j + kColWarps) * nc], fp[int64_t(j + kColWarps) * nc], s1);
        s2 = fma(ft[int64_t(j + 2 * kColWarps) * nc], fp[int64_t(j + 2 * kColWarps) * nc], s2);
        s3 = fma(ft[int64_t(j + 3 * kColWarps) * nc], fp[int64_t(j + 3 * kColWarps) * nc], s3);
      }
      for (; j < col; j += kColWarps) s0 = fma(ft[int64_t(j) * nc], fp[int64_t(j) * nc], s0);
      s = (s0 + s1) + (s2 + s3);
    }
    part[(0 * kColWarps + warp) * 32 + lane] = aL;
    part[(1 * kColWarps + warp) * 32 + lane] = aN;
    part[(2 * kColWarps + warp) * 32 + lane] = s;
    __syncthreads();
    if (warp == 0 && valid) {
      aL = aN = s = 0.0;
      for (int q = 0; q < kColWarps; ++q) {
        aL += part[(0 * kColWarps + q) * 32 + lane];
        aN += part[(1 * kColWarps + q) * 32 + lane];
        s += part[(2 * kColWarps + q) * 32 + lane];
      }
      const double m = w * (aL * (aL + 2.0 * aN));
      double v = (m - s) / sq;
      if (t == tp) v = sq;
      fac[int64_t(col) * nc + t] = v;
      const double left = (t == tp) ? 0.0 : d[t] - v * v;
      d[t] = left;
      dmax = fmax(dmax, left);
    }
    __syncthreads();
  }
  if (warp == 0) {
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0 && dmax > 0.0) atomicMax(&st->lmax[l], (unsigned long long)__double_as_longlong(dmax));
  }
}

// ---------------------------------------------------------------- speculative blocks
//
// A block of the greedy loop first guesses a set S of up to s points that are
// likely to be the next pivots (the largest local maxima of the residual on
// the grids) and computes the factor columns they would produce with
// tensor-core products over all candidates,
//   B[j][t] = w M(t, S_j) - sum_{k < kb} L[t,k] L[S_j,k]        (kb = columns so far).
// Greedy steps within S then need no other candidate: one CTA (k_blk_greedy)
// takes up to m of them on S's own residuals, finishing each column at the
// members of S from B with the columns added inside the block,
//   L[t,col] = (B[pos(p)][t] - sum_{kb <= k < col} L[t,k] L[p,k]) / sqrt(d_p).
// k_blk_apply then finishes the same columns at every candidate in the same
// arithmetic and looks for the first step at which some candidate's residual
// shows that the step was not the greedy one: its residual is above the step's
// maximum, or inside the step's tie window with a smaller index.  The steps
// before that one are exactly the ordinary greedy steps, the argmax over ALL
// candidates' residuals with the same tie rule; k_blk_commit takes them over.
// No step waits for the whole chip: three launches serve up to s steps, where
// a cooperative launch with two grid barriers per step took 13 us a step on one
// cell and 20 us on the 2x2x2 workload.  Per block: one cell 182 -> 94 us, 2x2x2
// 860 -> 434 us, the digits of the new columns included.

constexpr int kMaxSet = 256;  // options.select_block's limit

struct StepRec {
  double dp, dmax;  // the pivot's residual, the largest residual
  int idx;          // pivot: index over all candidates
  int t, pos;       // candidate in its level; row of B
  int lev;
};

// One round of a block: tried steps, their entries in the block's earlier
// columns, and the first step that failed.
struct BlkRound {
  int nsteps;
  int jstar;  // steps [0, jstar) are accepted
  int nl[ISDF_MAX_LEVELS];
  int list[ISDF_MAX_LEVELS][kMaxSet];  // steps of each level in order
  StepRec rec[kMaxSet];
  float2 lp[kMaxSet][kMaxSet];         // lp[step][q] = L[p_step, kb + q], double-float
};

struct BlkParams {
  SelParams P;
  const double* bm[ISDF_MAX_LEVELS];  // [s_l][nc_l]
  float2* bdf[ISDF_MAX_LEVELS];       // [s][nc_l] the block's columns so far, double-float
  const int* sidx;                    // S in ascending candidate order: index over all candidates
  const int* st;                      // and position in its level
  const int* scount;                  // per level, then in all
  int kb[ISDF_MAX_LEVELS];            // factor columns when S was chosen
  int kl[ISDF_MAX_LEVELS];            // factor columns now
  int k;                              // pivots now
  int64_t boff[ISDF_MAX_LEVELS + 1];  // blocks of kApply candidates per level
  const int* fexp[ISDF_MAX_LEVELS];   // fixed row scales and digit planes of the factor columns
  void* ftiles[ISDF_MAX_LEVELS];
  int64_t fkst[ISDF_MAX_LEVELS];
};

// Order-preserving key of a residual value: its bits when positive, else 0
// (integer operations only).
__device__ __forceinline__ unsigned long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 ? (unsigned long long)b : 0ull;
}

// Column entry of a block step for one candidate:
//   v = (b - sum_q F_q lp_q) / sqrt(d_p),
// F_q the block's earlier columns at this candidate (stride nc) and lp_q at
// the pivot, all double-float; the products' errors and the partial sums'
// rounding errors are gathered in one FP32 word.  FP32 pipes only.
__device__ __forceinline__ DF blk_col_df(const float2* __restrict__ fq, int64_t nc, int nbk, const DF* lpd, double b,
                                         DF inv_sq) {
  float ah = 0.0f, al = 0.0f;
  int q = 0;
  for (; q + 4 <= nbk; q += 4) {
    float2 c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) c[u] = __ldcg(fq + int64_t(q + u) * nc);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const DF l = lpd[q + u];
      const float pr = __fmul_rn(c[u].x, l.hi);
      float e = __fmaf_rn(c[u].x, l.hi, -pr);
      e = __fmaf_rn(c[u].x, l.lo, e);
      e = __fmaf_rn(c[u].y, l.hi, e);
      const DF t = two_sum(ah, pr);
      ah = t.hi;
      al = __fadd_rn(al, __fadd_rn(t.lo, e));
    }
  }
  for (; q < nbk; ++q) {
    const float2 c = __ldcg(fq + int64_t(q) * nc);
    const DF l = lpd[q];
    const float pr = __fmul_rn(c.x, l.hi);
    float e = __fmaf_rn(c.x, l.hi, -pr);
    e = __fmaf_rn(c.x, l.lo, e);
    e = __fmaf_rn(c.y, l.hi, e);
    const DF t = two_sum(ah, pr);
    ah = t.hi;
    al = __fadd_rn(al, __fadd_rn(t.lo, e));
  }
  return df_mul(df_sub(df_from_double(b), two_sum(ah, al)), inv_sq);
}

struct LmParams {
  const double* d;
  int64_t ntot;
  int nlev;
  int64_t coff[ISDF_MAX_LEVELS + 1];
  const int* cidx[ISDF_MAX_LEVELS];  // candidate -> grid index (nullptr: identity)
  const int* gpos[ISDF_MAX_LEVELS];  // grid index -> candidate (-1: none; nullptr: identity)
  int n[ISDF_MAX_LEVELS][3];
};

// d at the 6 periodic grid neighbours of candidate i (non-candidates count 0)
__device__ __forceinline__ bool is_local_max(const LmParams& Q, int64_t i) {
  const double v = Q.d[i];
  if (!(v > 0.0)) return false;
  int l = 0;
  while (l + 1 < Q.nlev && i >= Q.coff[l + 1]) ++l;
  const int64_t t = i - Q.coff[l];
  const int64_t g = Q.cidx[l] ? Q.cidx[l][t] : t;
  const int nx = Q.n[l][0], ny = Q.n[l][1], nz = Q.n[l][2];
  const int x = int(g % nx), y = int((g / nx) % ny), z = int(g / (int64_t(nx) * ny));
  const double* dl = Q.d + Q.coff[l];
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    int xx = x, yy = y, zz = z;
    if (a == 0) xx = x + 1 == nx ? 0 : x + 1;
    if (a == 1) xx = x == 0 ? nx - 1 : x - 1;
    if (a == 2) yy = y + 1 == ny ? 0 : y + 1;
    if (a == 3) yy = y == 0 ? ny - 1 : y - 1;
    if (a == 4) zz = z + 1 == nz ? 0 : z + 1;
    if (a == 5) zz = z == 0 ? nz - 1 : z - 1;
    const int64_t gg = xx + int64_t(nx) * (yy + int64_t(ny) * zz);
    const int64_t tt = Q.gpos[l] ? int64_t(Q.gpos[l][gg]) : gg;
    if (tt >= 0 && dl[tt] > v) return false;
  }
  return true;
}

// append the local maxima to a list (any order; k_top_s sorts what it keeps)
__global__ void __launch_bounds__(256) k_lm_list(LmParams Q, int* __restrict__ list, int* __restrict__ n) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool f = i < Q.ntot && is_local_max(Q, i);
  const unsigned b = __ballot_sync(0xffffffffu, f);
  if (!b) return;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0) base = atomicAdd(n, __popc(b));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (f) list[base + __popc(b & ((1u << lane) - 1u))] = int(i);
}

// The s largest residuals of the list (ties to the smallest index), by an
// 8-bit radix select on the bit patterns (d > 0 orders like its bits), then on
// the indices of those equal to the last one kept.  Writes S in ascending
// candidate order: sidx (concatenated index), sg (grid index), st (position in
// its level), per-level counts.  One CTA, bound by the latency of its passes
// over the list: the bins are searched by one warp (a thread walking 256 bins
// cost 4 us a pass, 39 us in all on one cell's lists; now 12).
struct TopSOut {
  int* sidx;
  int* sg;
  int* st;
  int* scount;  // [ISDF_MAX_LEVELS + 1]: per-level counts, then the total
};
constexpr int kTopKeys = 4096;  // keys kept in shared memory (longer lists are read from global memory)

// Highest bin b (from the top) with count(bins > b) + above < want <= count(bins >= b) + above; one warp.
__device__ __forceinline__ void pick_bin(const int* hist, int above, int want, int lane, int* bin, int* gt) {
  int c[8], tot = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) tot += c[q] = hist[255 - (lane * 8 + q)];
  int pre = tot;  // inclusive prefix over lanes (lane 0: the top bins)
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, pre, o);
    if (lane >= o) pre += x;
  }
  int acc = above + pre - tot;
  if (acc < want && want <= acc + tot) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (acc < want && want <= acc + c[q]) *bin = 255 - (lane * 8 + q), *gt = acc;
      acc += c[q];
    }
  }
}

__global__ void __launch_bounds__(1024) k_top_s(LmParams Q, const int* __restrict__ list, const int* __restrict__ nlist,
                                                int smax, TopSOut O) {
  __shared__ unsigned long long skey[kTopKeys];
  __shared__ int hist[256];
  __shared__ int bin_sh, gt_sh, kept;
  __shared__ int sel[kMaxSet];
  __shared__ int lcount[ISDF_MAX_LEVELS];
  const int n = *nlist, tid = threadIdx.x, lane = tid & 31;
  const int want = n < smax ? n : smax;
  if (tid == 0) kept = 0;
  if (tid < ISDF_MAX_LEVELS) lcount[tid] = 0;
  auto load_key = [&](int i) { return (unsigned long long)__double_as_longlong(Q.d[list[i]]); };
  for (int i = tid; i < n && i < kTopKeys; i += 1024) skey[i] = load_key(i);
  __syncthreads();
  auto key = [&](int i) { return i < kTopKeys ? skey[i] : load_key(i); };
  unsigned long long T = 0ull, mask = 0ull;
  unsigned int tie = 0xffffffffu;  // among keys equal to T: indices up to tie
  if (want > 0 && want < n) {
    int above = 0;
    for (int pass = 0; pass < 12; ++pass) {
      // passes 0..7: the threshold key; 8..11: the largest index kept among its equals
      const bool on_key = pass < 8;
      const int shift = on_key ? 56 - 8 * pass : 88 - 8 * pass;
      if (pass == 8) tie = 0u, mask = 0ull;
      if (tid < 256) hist[tid] = 0;
      __syncthreads();
      for (int i = tid; i < n; i += 1024) {
        const unsigned long long k = key(i);
        if (on_key) {
          if ((k & mask) == T) atomicAdd(&hist[(k >> shift) & 255], 1);
        } else if (k == T) {
          const unsigned int x = ~(unsigned int)list[i];  // smallest index first
          if ((x & (unsigned int)mask) == tie) atomicAdd(&hist[(x >> shift) & 255], 1);
        }
      }
      __syncthreads();
      if (tid < 32) pick_bin(hist, above, want, lane, &bin_sh, &gt_sh);
      __syncthreads();
      above = gt_sh;
      mask |= 255ull << shift;
      if (on_key) T |= (unsigned long long)bin_sh << shift;
      else tie |= (unsigned int)bin_sh << shift;
      // all of the keys equal to T are wanted: no choice among them
      if (pass == 7 && above + hist[bin_sh] == want) {
        tie = 0u;
        break;
      }
      __syncthreads();
    }
  } else {
    tie = 0u;
  }
  __syncthreads();
  for (int i = tid; i < n; i += 1024) {
    const unsigned long long k = key(i);
    const int idx = list[i];
    if (k > T || (k == T && ~(unsigned int)idx >= tie)) sel[atomicAdd(&kept, 1)] = idx;
  }
  __syncthreads();
  const int total = kept;  // = want
  if (tid < total) {
    const int idx = sel[tid];
    int rank = 0;
    for (int i = 0; i < total; ++i) rank += sel[i] < idx;
    int l = 0;
    while (l + 1 < Q.nlev && idx >= Q.coff[l + 1]) ++l;
    const int64_t t = idx - Q.coff[l];
    O.sidx[rank] = idx;
    O.st[rank] = int(t);
    O.sg[rank] = Q.cidx[l] ? Q.cidx[l][t] : int(t);
    atomicAdd(&lcount[l], 1);
  }
  __syncthreads();
  if (tid == 0) {
    for (int l = 0; l < ISDF_MAX_LEVELS; ++l) O.scount[l] = l < Q.nlev ? lcount[l] : 0;
    O.scount[ISDF_MAX_LEVELS] = total;
  }
}

// Fixed row scales of the factor columns: |L[c][k]| <= sqrt(d0_c)
__global__ void k_fac_exps(const double* __restrict__ d0c, int64_t nc, int64_t npad, int* __restrict__ exps) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= npad) return;
  int e = 0;
  if (t < nc && d0c[t] > 0.0) frexp(sqrt(d0c[t]) * (1.0 + 0x1p-20), &e);
  exps[t] = e;
}

// before an ordinary step between two blocks
__global__ void k_step_begin(SelState* st) {
  if (threadIdx.x != 0) return;
  st->done = st->final_ ? 1 : 0;
  st->skip = 1;
  for (int l = 0; l < ISDF_MAX_LEVELS; ++l) st->lmax[l] = 0ull;
  st->first = ULLONG_MAX;
  st->arrived = 0u;
}

// Largest of a warp's 64-bit keys: two 32-bit warp reductions.
__device__ __forceinline__ unsigned long long warp_max64(unsigned long long k) {
  const unsigned hi = unsigned(k >> 32), h = __reduce_max_sync(0xffffffffu, hi);
  const unsigned l = __reduce_max_sync(0xffffffffu, hi == h ? unsigned(k) : 0u);
  return (unsigned long long)h << 32 | l;
}

// The tie threshold of a step: d >= thr and d > 0  <=>  key(d) >= tie_key.
__device__ __forceinline__ unsigned long long tie_key(const SelParams& P, double dmax, double d0) {
  return max(dkey(dmax - fmax(P.tie_rel * dmax, P.tie_abs * d0)), 1ull);
}

// Up to m greedy steps among the members of S, one thread per member.  A step
// is a chain of two block syncs, the members' dots over the block's earlier
// columns (double-float, the arithmetic of k_blk_apply) and two FP64
// operations: the FP64 unit takes hundreds of cycles for a chain of a few
// operations, so the reciprocal root is a double-float one, the tie window is
// first tested against an integer bound from below (one member above it is
// the pivot whatever the exact threshold is), and square roots and thresholds
// of the record are left to k_blk_apply.  With `gcols` null the columns and B at
// S x S are in shared memory ([s][nwork] each), so no step waits for L2; else
// (more members than fit) the columns are in gcols and B is read in place.
// (With the FP64 scalars in the chain and four syncs a step took 2.6 us.)
__global__ void __launch_bounds__(kMaxSet) k_blk_greedy(BlkParams B, SelState* st, BlkRound* R, int m, int smax,
                                                        float2* __restrict__ gcols) {
  extern __shared__ double sm_greedy[];
  __shared__ unsigned long long wmax[kMaxSet / 32];
  __shared__ int wfirst[kMaxSet / 32], wcount[kMaxSet / 32];
  __shared__ unsigned long long thr_sh;
  __shared__ double dmem[kMaxSet];
  const SelParams& P = B.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwork = blockDim.x, nwarp = nwork >> 5;
  int begin[ISDF_MAX_LEVELS + 1] = {0};  // members of level l: [begin[l], begin[l + 1])
#pragma unroll
  for (int l = 0; l < ISDF_MAX_LEVELS; ++l) begin[l + 1] = begin[l] + B.scount[l];
  const int total = begin[ISDF_MAX_LEVELS];
  int lev = 0, mfirst = 0, mlast = begin[1];  // this member's level and its range
#pragma unroll
  for (int l = 1; l < ISDF_MAX_LEVELS; ++l)
    if (l < P.nlev && tid >= begin[l]) lev = l, mfirst = begin[l], mlast = begin[l + 1];
  const bool mine = tid < total;
  const int64_t nc = P.nc[lev];
  const int64_t t = mine ? B.st[tid] : 0;
  const int gidx = mine ? B.sidx[tid] : 0;
  double* bss = sm_greedy;  // B[member p][this thread] at p * nwork + tid
  float2* cols = gcols ? gcols : reinterpret_cast<float2*>(sm_greedy + int64_t(smax) * nwork);  // q * nwork + tid
  double d = mine ? P.d[gidx] : 0.0;
  if (!gcols && mine) {
    const double* b = B.bm[lev] + t;
#pragma unroll 8
    for (int i = mfirst; i < mlast; ++i) bss[i * nwork + tid] = __ldcg(b + int64_t(i - mfirst) * nc);
  }
  unsigned long long key = mine ? dkey(d) : 0ull;
  int nq[ISDF_MAX_LEVELS];  // columns in the block, per level (the same in every thread)
  int nstep[ISDF_MAX_LEVELS] = {0, 0, 0, 0};
  int mynq = 0;
#pragma unroll
  for (int l = 0; l < ISDF_MAX_LEVELS; ++l) {
    nq[l] = B.kl[l] - B.kb[l];
    if (l == lev) mynq = nq[l];
  }
  if (mine)
    for (int q = 0; q < mynq; ++q) cols[q * nwork + tid] = __ldcg(B.bdf[lev] + int64_t(q) * nc + t);
  if (mine) dmem[tid] = d;
  double d0 = st->d0;
  // binary exponents: tie_rel < 2^(e_rel + 1), tie_abs d0 < 2^(e_abs + 1) 2^-1023
  const int e_rel = int(dkey(P.tie_rel) >> 52) - 1023;
  int e_abs = int(dkey(P.tie_abs * d0) >> 52);
  int j = 0;
  for (; j < m; ++j) {
    // ---- the largest residual
    const unsigned long long wk = warp_max64(key);
    if (lane == 0) wmax[warp] = wk;
    __syncthreads();
    const unsigned long long mk = warp_max64(lane < nwarp ? wmax[lane] : 0ull);
    const double dmax = __longlong_as_double((long long)mk);
    const int k = B.k + j;
    // no further pivot: the next block's set, or an ordinary step, decides what that means
    if (k >= P.nip || mk == 0ull) break;
    if ((mk >> 52) == 0x7FFull) break;  // infinite: no threshold, so no member would be found below
    if (P.tol > 0.0 && k > 0 && dmax < P.tol * d0) break;
    if (k == 0) {
      d0 = dmax;
      e_abs = int(dkey(P.tie_abs * d0) >> 52);
      if (tid == 0) {
        st->d0 = dmax;
        st->t0 = globaltimer();
      }
    }
    // ---- the smallest index within the tie window (members are in index
    // order).  A relative distance x <= 1/4 below dmax is less than x 2^54 keys;
    // x is bounded by the power of two above it.
    const int sh = 55 + max(e_rel, e_abs - int(mk >> 52));
    const bool hit = key >= ((sh < 53 && (mk >> 54)) ? mk - (1ull << max(sh, 2)) : 1ull);
    unsigned b0 = __ballot_sync(0xffffffffu, hit);
    if (lane == 0) {
      wfirst[warp] = b0 ? warp * 32 + __ffs(int(b0)) - 1 : INT_MAX;
      wcount[warp] = __popc(b0);
    }
    __syncthreads();
    int p = __reduce_min_sync(0xffffffffu, lane < nwarp ? wfirst[lane] : INT_MAX);
    const int nhit = __reduce_add_sync(0xffffffffu, lane < nwarp ? unsigned(wcount[lane]) : 0u);
    if (nhit > 1) {  // more than one member near the maximum: the exact window
      if (tid == 0) thr_sh = tie_key(P, dmax, d0);
      __syncthreads();
      b0 = __ballot_sync(0xffffffffu, key >= thr_sh);
      if (lane == 0) wfirst[warp] = b0 ? warp * 32 + __ffs(int(b0)) - 1 : INT_MAX;
      __syncthreads();
      p = __reduce_min_sync(0xffffffffu, lane < nwarp ? wfirst[lane] : INT_MAX);
    }
    int pl = 0, pfirst = 0, q = nq[0], c = nstep[0];
#pragma unroll
    for (int l = 1; l < ISDF_MAX_LEVELS; ++l)
      if (l < P.nlev && p >= begin[l]) pl = l, pfirst = begin[l], q = nq[l], c = nstep[l];
    // ---- its column at the members of its level
    const double dp = dmem[p];
    for (int i = tid; i < q; i += nwork) R->lp[j][i] = cols[i * nwork + p];
    if (tid == p) {
      StepRec& rec = R->rec[j];
      rec.dp = dp;
      rec.dmax = dmax;
      rec.idx = gidx;
      rec.t = int(t);
      rec.pos = p - pfirst;
      rec.lev = pl;
      R->list[pl][c] = j;
      key = 0ull;
    } else if (mine && lev == pl && key) {
      const double b = gcols ? __ldcg(B.bm[pl] + int64_t(p - pfirst) * nc + t) : bss[p * nwork + tid];
      float ah = 0.0f, al = 0.0f;
#pragma unroll 4
      for (int i = 0; i < q; ++i) {
        const float2 x = cols[i * nwork + tid], l = cols[i * nwork + p];
        const float pr = __fmul_rn(x.x, l.x);
        float e = __fmaf_rn(x.x, l.x, -pr);
        e = __fmaf_rn(x.x, l.y, e);
        e = __fmaf_rn(x.y, l.x, e);
        const DF s = two_sum(ah, pr);
        ah = s.hi;
        al = __fadd_rn(al, __fadd_rn(s.lo, e));
      }
      const DF v = df_mul(df_sub(df_from_double(b), two_sum(ah, al)), df_rsqrt(dp));
      cols[q * nwork + tid] = make_float2(v.hi, v.lo);
      const double vd = df_to_double(v);
      d = fma(-vd, vd, d);
      key = dkey(d);
      dmem[tid] = d;
    }
#pragma unroll
    for (int l = 0; l < ISDF_MAX_LEVELS; ++l)
      if (l == pl) ++nq[l], ++nstep[l];
  }
  if (tid == 0) {
    R->nsteps = j;
    R->jstar = j;
#pragma unroll
    for (int l = 0; l < ISDF_MAX_LEVELS; ++l) R->nl[l] = nstep[l];
  }
}

// The tried columns at every candidate, and the first step that some candidate
// shows not to be the greedy one (atomicMin into jstar; threads stop at it).
// A candidate's entry of a step needs its entries of the level's earlier
// columns in the block (double-float, from L1/L2), so one thread walks one
// candidate through all steps of its level.
constexpr int kApply = 128;
__global__ void __launch_bounds__(kApply) k_blk_apply(BlkParams B, const SelState* st, BlkRound* R) {
  const SelParams& P = B.P;
  __shared__ unsigned long long dmax_s[kMaxSet], thr_s[kMaxSet];
  __shared__ int idx_s[kMaxSet], list_s[kMaxSet], pos_s[kMaxSet], t_s[kMaxSet];
  __shared__ DF inv_s[kMaxSet], lp_s[2][kMaxSet];
  __shared__ double sq_s[kMaxSet];
  const int tid = threadIdx.x;
  int l = 0;
  while (l + 1 < P.nlev && int64_t(blockIdx.x) >= B.boff[l + 1]) ++l;
  const int64_t nc = P.nc[l], t = (int64_t(blockIdx.x) - B.boff[l]) * kApply + tid;
  const bool live = t < nc;
  const int ns = R->nsteps, nl = R->nl[l], q0 = B.kl[l] - B.kb[l];
  for (int i = tid; i < ns; i += kApply) {
    const StepRec& r = R->rec[i];
    dmax_s[i] = dkey(r.dmax);
    thr_s[i] = tie_key(P, r.dmax, st->d0);
    idx_s[i] = r.idx;
  }
  for (int k = tid; k < nl; k += kApply) {
    const int i = R->list[l][k];
    const StepRec& r = R->rec[i];
    list_s[k] = i;
    pos_s[k] = r.pos;
    t_s[k] = r.t;
    inv_s[k] = df_rsqrt(r.dp);
    sq_s[k] = root64(r.dp).s;
  }
  auto stage = [&](int k) {  // lp of the level's step k
    for (int i = tid; i < q0 + k; i += kApply) {
      const float2 c = R->lp[list_s[k]][i];
      lp_s[k & 1][i] = {c.x, c.y};
    }
  };
  __syncthreads();
  if (nl > 0) stage(0);
  const int64_t gi = P.coff[l] + t;
  double d = live ? P.d[gi] : 0.0;
  unsigned long long key = dkey(d);
  bool on = live;
  int from = 0;  // first step not checked yet
  float2* bdf = B.bdf[l] + t;
  // the residual stands still over steps [from, to]: the step maxima fall, so
  // only the last threshold has to be looked at when it is not reached
  auto check = [&](int to) {
    if (!on || to < from) return;
    if (key >= thr_s[to])
      for (int i = from; i <= to; ++i)
        if (key > dmax_s[i] || (key >= thr_s[i] && gi < idx_s[i])) {
          atomicMin(&R->jstar, i);
          on = false;
          break;
        }
    from = to + 1;
  };
  double bnext = (on && nl > 0) ? B.bm[l][int64_t(pos_s[0]) * nc + t] : 0.0;
  for (int k = 0; k < nl; ++k) {
    __syncthreads();
    const int i = list_s[k];
    const int js = *(volatile int*)&R->jstar;
    if (i >= js) {  // this step is lost; the ones before it still need this candidate's word
      check(js - 1);
      on = false;
    }
    if (!__syncthreads_or(on)) return;
    if (k + 1 < nl) stage(k + 1);
    check(i);
    if (!on) continue;
    const double b = bnext;
    if (k + 1 < nl) bnext = B.bm[l][int64_t(pos_s[k + 1]) * nc + t];
    const bool pivot = t == t_s[k];
    const double sq = sq_s[k];
    const DF v = pivot ? df_from_double(sq) : blk_col_df(bdf, nc, q0 + k, lp_s[k & 1], b, inv_s[k]);
    const double vd = pivot ? sq : df_to_double(v);
    P.fac[l][int64_t(B.kl[l] + k) * nc + t] = vd;
    bdf[int64_t(q0 + k) * nc] = make_float2(v.hi, v.lo);
    if (pivot) {
      key = 0ull;  // taken: it takes no part in later steps, but its row does
      d = 0.0;
    } else if (key) {
      d = fma(-vd, vd, d);
      key = dkey(d);
    }
  }
  if (ns > 0) check(ns - 1);
}

// Accept steps [0, jstar): residuals, the digits of the new columns (whole
// groups of 8, from the first one touched) and the state record.
__global__ void __launch_bounds__(kApply) k_blk_commit(BlkParams B, BlkRound* R, SelState* st) {
  const SelParams& P = B.P;
  const int tid = threadIdx.x, js = R->jstar;
  int l = 0;
  while (l + 1 < P.nlev && int64_t(blockIdx.x) >= B.boff[l + 1]) ++l;
  if (blockIdx.x == 0) {
    for (int i = tid; i < js; i += kApply) {
      const StepRec& r = R->rec[i];
      const long long g = P.cidx[r.lev] ? P.cidx[r.lev][r.t] : r.t;
      P.piv[B.k + i] = ((long long)r.lev << kPivShift) | g;
      P.dval[B.k + i] = r.dp;
    }
    if (tid == 0) {
      st->bsteps = js;
      for (int a = 0; a < P.nlev; ++a) st->members[a] = B.scount[a];
      st->k = B.k + js;
      for (int a = 0; a < P.nlev; ++a) {
        int c = 0;
        while (c < R->nl[a] && R->list[a][c] < js) ++c;
        st->kl[a] = B.kl[a] + c;
      }
      if (js > 0) st->dp = R->rec[js - 1].dp;
      if (js > 0 && P.timeout_ns && globaltimer() - st->t0 > P.timeout_ns) {
        st->err = ISDF_ERR_TIMEOUT;
        st->final_ = 1;
      }
    }
  }
  const int64_t nc = P.nc[l], t = (int64_t(blockIdx.x) - B.boff[l]) * kApply + tid;
  int na = 0;
  while (na < R->nl[l] && R->list[l][na] < js) ++na;
  if (t >= nc || na == 0) return;
  const double* fac = P.fac[l] + t;
  const int c0 = B.kl[l], c1 = c0 + na;
  double d = P.d[P.coff[l] + t];
  if (dkey(d)) {
    for (int k = 0; k < na; ++k) {
      const double v = fac[int64_t(c0 + k) * nc];
      d = R->rec[R->list[l][k]].t == t ? 0.0 : fma(-v, v, d);
      if (!dkey(d)) break;
    }
    P.d[P.coff[l] + t] = d;
  }
  oz_append_row(fac, nc, c0, c1, B.fexp[l][t], t, B.fkst[l], B.ftiles[l]);
}

}  // namespace

namespace {

constexpr unsigned kColBlocks = 152 * 6;  // fallback grid if the occupancy query fails

// Limits of dynamic shared memory.  They belong to the kernel, not to a plan:
// every selection sets the same value, so that no thread lowers it under
// another's launches.
constexpr size_t kColSmem = 227 * 1024;     // k_sel_col, when a plan needs more than 48 KB
constexpr size_t kGreedySmem = 216 * 1024;  // k_blk_greedy; more members than fit work in global memory

// One greedy run over the given candidates (cidx[l] == nullptr: all points).
isdf_status select_loop(Plan* p, int nip, double tol, const double* d0full, int* const* cidx, const int64_t* nc,
                        int* nfound, int* kl_out) {
  cudaStream_t s = p->stream;
  isdf_status st;
  SelParams P{};
  P.nlev = p->nlev;
  P.coff[0] = 0;
  int nGmax = 1;
  for (int l = 0; l < p->nlev; ++l) {
    P.coff[l + 1] = P.coff[l] + nc[l];
    P.cidx[l] = cidx[l];
    P.nc[l] = nc[l];
  }
  P.ntot = P.coff[p->nlev];
  dfree(p->d_diag);
  p->d_diag = nullptr;
  if ((st = dalloc_t(p, &p->d_diag, size_t(std::max<int64_t>(P.ntot, 1)), "residual diagonal"))) return st;
  P.d = p->d_diag;
  for (int l = 0; l < p->nlev; ++l) {
    Level& lv = p->lev[l];
    dfree(lv.fac);
    lv.fac = nullptr;
    lv.fac_cap = std::min<int64_t>(nip, nc[l]);
    if ((st = dalloc_t(p, &lv.fac, size_t(std::max<int64_t>(lv.fac_cap * nc[l], 1)), "selection factor columns")))
      return st;
    P.fac[l] = lv.fac;
    P.phi[l] = lv.phi;
    P.ng[l] = lv.ng;
    P.nL[l] = lv.nL;
    P.nG[l] = lv.nG;
    P.w[l] = lv.w;
    nGmax = std::max(nGmax, lv.nG);
    if (nc[l]) {
      k_gather_diag<<<unsigned((nc[l] + 255) / 256), 256, 0, s>>>(d0full + p->off[l], cidx[l], nc[l],
                                                                  p->d_diag + P.coff[l]);
      count_launches(1);
    }
  }
  P.piv = p->d_piv;
  P.dval = p->d_dval;
  P.nip = nip;
  P.tol = tol;
  P.tie_rel = p->opt.tie_rel;
  P.tie_abs = p->opt.tie_abs;
  P.timeout_ns = (unsigned long long)p->opt.timeout_ms * 1000000ull;
  SelState h{};
  h.first = ULLONG_MAX;
  h.skip = 1;
  if ((st = cuda_check(p, cudaMemcpyAsync(p->d_selstate, &h, sizeof(h), cudaMemcpyHostToDevice, s), "state init")))
    return st;
  SelState* dst = static_cast<SelState*>(p->d_selstate);
  const size_t smem = sizeof(double) * (size_t((nGmax + 1) & ~1) + 3 * kColWarps * 32);
  if (smem > 48 * 1024) {
    if ((st = cuda_check(p, cudaFuncSetAttribute(k_sel_col, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kColSmem)),
                         "smem attribute")))
      return st;
  }
  // one wave of resident blocks: grid-striding then splits the groups evenly
  int dev = 0, nsm = 152, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sel_col, 32 * kColWarps, smem);
  const unsigned red_blocks = sel_blocks(P.ntot, nsm);
  const unsigned col_blocks = per_sm > 0 ? unsigned(per_sm * nsm) : kColBlocks;
  k_sel_max<<<dim3(red_blocks, unsigned(P.nlev)), 256, 0, s>>>(P, dst);
  count_launches(1);
  auto one_step = [&]() {
    k_sel_first<<<red_blocks, 256, 0, s>>>(P, dst);
    k_sel_col<<<col_blocks, 256, smem, s>>>(P, dst);
  };
  // Capture a chunk of steps into a graph (not possible on the legacy stream).
  const int chunk = 32;
  bool graphed = false;
  Prof* loop_prof = new Prof(p, "select_loop", 0.0, "flop", 2ll * nip);
  if (s != nullptr && nip >= chunk) {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      for (int i = 0; i < chunk; ++i) one_step();
      if (cudaStreamEndCapture(s, &graph) == cudaSuccess && graph &&
          cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess) {
        graphed = true;
        const int full = nip / chunk;
        for (int c = 0; c < full; ++c) cudaGraphLaunch(exec, s);
        for (int i = full * chunk; i < nip; ++i) one_step();
      }
      if (exec) {
        cudaStreamSynchronize(s);
        cudaGraphExecDestroy(exec);
      }
      if (graph) cudaGraphDestroy(graph);
    }
    cudaGetLastError();  // a failed capture leaves a sticky-free error; clear it
  }
  if (!graphed)
    for (int i = 0; i < nip; ++i) one_step();
  delete loop_prof;  // records the end event; work is filled in below
  if ((st = cuda_check(p, cudaGetLastError(), "selection kernels"))) return st;
  if ((st = cuda_check(p, cudaMemcpyAsync(&h, p->d_selstate, sizeof(h), cudaMemcpyDeviceToHost, s), "state copy")))
    return st;
  if ((st = cuda_check(p, cudaStreamSynchronize(s), "selection"))) return st;
  *nfound = h.k;
  for (int l = 0; l < p->nlev; ++l) kl_out[l] = h.kl[l];
  if (p->opt.profile && !p->pend.empty() && p->pend.back().name == "select_loop") {
    // algorithmic flops: step c on level l costs 2 (nG + c) n_cand (M column
    // and the factor-row dot product)
    double work = 0.0;
    for (int l = 0; l < p->nlev; ++l) {
      const double k = h.kl[l], n = double(nc[l]), nG = p->lev[l].nG;
      work += 2.0 * n * (nG * k + 0.5 * k * (k - 1.0));
    }
    p->pend.back().work = work;
  }
  for (int l = 0; l < p->nlev; ++l) {  // factor columns are not needed after selection
    dfree(p->lev[l].fac);
    p->lev[l].fac = nullptr;
  }
  if (h.err == ISDF_ERR_TIMEOUT) return fail(p, ISDF_ERR_TIMEOUT, "selection loop exceeded options.timeout_ms");
  return ISDF_OK;
}

__global__ void k_scatter_pos(const int* __restrict__ cidx, int64_t nc, int* __restrict__ gpos) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < nc) gpos[cidx[t]] = int(t);
}

// out[j] = in ? in[keep[j]] : keep[j]  (candidate grid indices after compaction)
__global__ void k_map_idx(const int* __restrict__ in, const int* __restrict__ keep, int64_t n, int* __restrict__ out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < n) out[t] = in ? in[keep[t]] : keep[t];
}

// fac_new[c][j] = fac_old[c][keep[j]] for the first ncol columns
__global__ void k_gather_cols(const double* __restrict__ fo, int64_t no, const int* __restrict__ keep, int64_t nn,
                              int64_t ncol, double* __restrict__ fn) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= nn * ncol) return;
  const int64_t c = e / nn, j = e % nn;
  fn[e] = fo[c * no + keep[j]];
}

constexpr int kSlices = 8;  // FP64-grade sliced products for the selection

// Speculative-block form of select_loop (same result: every pivot is the
// greedy one).  Per block: S from the residual's local maxima, the columns of S
// at every candidate in one tensor-core launch, then rounds of greedy steps among
// the members of S (k_blk_greedy), verified at every candidate (k_blk_apply) and
// taken over up to the first step that failed (k_blk_commit).  A round that
// loses a step ends the block; if it accepted none, one ordinary step is taken.
// tau > 0: the candidates are the points with initial residual >= tau (the
// exact prefilter).  Residuals only shrink, so a candidate whose residual
// falls below tau can never be picked while every pivot value stays above
// tau plus the tie margin (the certificate select_run checks): between
// blocks such candidates are dropped and every candidate-side array is
// rebuilt for the rest, which changes no pivot and no column entry (rows
// are computed independently, ties go to the smallest grid index either
// way).  As soon as a pivot value breaks the certificate the attempt stops
// (*aborted) so that select_run can retry with a lower tau.
isdf_status select_loop_blocked(Plan* p, int nip, double tol, const double* d0full, int* const* cidx,
                                const int64_t* nc_in, int* nfound, int* kl_out, double tau, bool* aborted) {
  cudaStream_t s = p->stream;
  isdf_status st = ISDF_OK;
  const int smax = p->opt.select_block;
  const int nlev = p->nlev;
  *aborted = false;
  int64_t nc[ISDF_MAX_LEVELS] = {0, 0, 0, 0};
  for (int l = 0; l < nlev; ++l) nc[l] = nc_in[l];
  int* cur_cidx[ISDF_MAX_LEVELS] = {nullptr, nullptr, nullptr, nullptr};  // after compaction: owned here
  for (int l = 0; l < nlev; ++l) cur_cidx[l] = cidx[l];
  std::vector<int*> own_cidx;
  SelParams P{};
  P.nlev = nlev;
  P.coff[0] = 0;
  int nGmax = 1;
  for (int l = 0; l < nlev; ++l) {
    P.coff[l + 1] = P.coff[l] + nc[l];
    P.cidx[l] = cidx[l];
    P.nc[l] = nc[l];
  }
  P.ntot = P.coff[nlev];
  dfree(p->d_diag);
  p->d_diag = nullptr;
  if ((st = dalloc_t(p, &p->d_diag, size_t(std::max<int64_t>(P.ntot, 1)), "residual diagonal"))) return st;
  P.d = p->d_diag;

  struct LevBuf {
    OzOperand aL, aN, aF, bL, bN, bF;
    double* col = nullptr;  // B of the block [s_l][nc]
    float2* bdf = nullptr;  // the block's columns so far, double-float [s][nc]
    int* gpos = nullptr;
  } lb[ISDF_MAX_LEVELS];
  int *counts = nullptr, *nlist = nullptr, *list = nullptr, *sidx = nullptr, *sg = nullptr, *stp = nullptr,
      *scount = nullptr;
  BlkRound* round = nullptr;
  float2* gcols = nullptr;
  auto cleanup = [&]() {
    for (int* q : own_cidx) dfree(q);
    own_cidx.clear();
    for (int l = 0; l < nlev; ++l) {
      oz_free(lb[l].aL), oz_free(lb[l].aN), oz_free(lb[l].aF);
      oz_free(lb[l].bL), oz_free(lb[l].bN), oz_free(lb[l].bF);
      dfree(lb[l].col), dfree(lb[l].bdf), dfree(lb[l].gpos);
      dfree(p->lev[l].fac);
      p->lev[l].fac = nullptr;
    }
    dfree(counts), dfree(nlist), dfree(list), dfree(sidx), dfree(sg), dfree(stp), dfree(scount);
    dfree(round), dfree(gcols);
  };
  auto bail = [&](isdf_status r) {
    cleanup();
    return r;
  };

  // ---- set-up: residual, factor storage, candidate-side operands
  LmParams Q{};
  Q.d = P.d;
  Q.nlev = nlev;
  Q.ntot = P.ntot;
  for (int l = 0; l <= nlev; ++l) Q.coff[l] = P.coff[l];
  for (int l = 0; l < nlev; ++l) {
    Level& lv = p->lev[l];
    LevBuf& b = lb[l];
    dfree(lv.fac);
    lv.fac = nullptr;
    // factor storage starts at a quarter of nip and grows between blocks (a level rarely takes more)
    lv.fac_cap = std::min<int64_t>(std::min<int64_t>(nip, nc[l]), std::max<int64_t>(4 * int64_t(smax) + 1, nip / 4));
    if ((st = dalloc_t(p, &lv.fac, size_t(std::max<int64_t>(lv.fac_cap * nc[l], 1)), "selection factor columns")))
      return bail(st);
    P.fac[l] = lv.fac;
    P.phi[l] = lv.phi;
    P.ng[l] = lv.ng;
    P.nL[l] = lv.nL;
    P.nG[l] = lv.nG;
    P.w[l] = lv.w;
    nGmax = std::max(nGmax, lv.nG);
    Q.cidx[l] = cidx[l];
    for (int a = 0; a < 3; ++a) Q.n[l][a] = lv.n[a];
    if (!nc[l]) continue;
    k_gather_diag<<<unsigned((nc[l] + 255) / 256), 256, 0, s>>>(d0full + p->off[l], cidx[l], nc[l], p->d_diag + P.coff[l]);
    count_launches(1);
    if (cidx[l]) {
      if ((st = dalloc_t(p, &b.gpos, size_t(lv.ng), "grid-to-candidate map"))) return bail(st);
      cudaMemsetAsync(b.gpos, 0xFF, sizeof(int) * size_t(lv.ng), s);
      k_scatter_pos<<<unsigned((nc[l] + 255) / 256), 256, 0, s>>>(cidx[l], nc[l], b.gpos);
      count_launches(1);
    }
    Q.gpos[l] = b.gpos;
    const int bn = oz_bn(kSlices);
    if ((st = oz_alloc(p, b.aL, nc[l], std::max(lv.nL, 1), 128, kSlices, "selection slices")) ||
        (st = oz_alloc(p, b.bL, smax, std::max(lv.nL, 1), bn, kSlices, "selection slices")) ||
        (st = oz_alloc(p, b.aF, nc[l], lv.fac_cap, 128, kSlices, "selection slices")) ||
        (st = oz_alloc(p, b.bF, smax, lv.fac_cap, bn, kSlices, "selection slices")) ||
        (st = dalloc_t(p, &b.col, size_t(smax) * nc[l], "selection columns")) ||
        (st = dalloc_t(p, &b.bdf, size_t(smax) * nc[l], "selection columns")))
      return bail(st);
    if (lv.nN > 0 && ((st = oz_alloc(p, b.aN, nc[l], lv.nN, 128, kSlices, "selection slices")) ||
                      (st = oz_alloc(p, b.bN, smax, lv.nN, bn, kSlices, "selection slices"))))
      return bail(st);
    {
      Prof pr(p, "select_slice", 8.0 * double(nc[l]) * lv.nG, "byte", 4);
      if (lv.nL > 0) oz_slice_ex(lv.phi, 1, lv.ng, cidx[l], b.aL, 0, b.aL.nkt * (kOzBK / 8), false, s);
      if (lv.nN > 0)
        oz_slice_ex(lv.phi + int64_t(lv.nL) * lv.ng, 1, lv.ng, cidx[l], b.aN, 0, b.aN.nkt * (kOzBK / 8), false, s);
      // factor-column digits are written group by group as columns appear:
      // groups not yet written must read as zero
      cudaMemsetAsync(b.aF.tiles, 0, size_t(oz_tile_bytes(b.aF)), s);
      // factor rows are bounded by sqrt(d0): fixed scales, columns appended in place
      k_fac_exps<<<unsigned((b.aF.nrt * 128 + 255) / 256), 256, 0, s>>>(p->d_diag + P.coff[l], nc[l], b.aF.nrt * 128,
                                                                         b.aF.exps);
      count_launches(1);
    }
    b.aF.K = 0;
    b.aF.nkt = 0;
  }
  P.piv = p->d_piv;
  P.dval = p->d_dval;
  P.nip = nip;
  P.tol = tol;
  P.tie_rel = p->opt.tie_rel;
  P.tie_abs = p->opt.tie_abs;
  P.timeout_ns = (unsigned long long)p->opt.timeout_ms * 1000000ull;
  const int64_t nbk = (P.ntot + kCompactBlock - 1) / kCompactBlock;
  // B and the members' columns during the greedy steps: shared memory up to 108 members, else global
  const int gthreads = ((smax + 31) / 32) * 32;
  const size_t gsmem = 2 * sizeof(double) * size_t(gthreads) * smax;
  const bool gshared = gsmem <= kGreedySmem;
  if ((st = dalloc_t(p, &counts, size_t(std::max<int64_t>(nbk, 1)), "block counts")) ||
      (st = dalloc_t(p, &nlist, 1, "list size")) ||
      (st = dalloc_t(p, &list, size_t(std::max<int64_t>(P.ntot, 1)), "local maxima")) ||
      (st = dalloc_t(p, &sidx, size_t(smax), "speculative set")) || (st = dalloc_t(p, &sg, size_t(smax), "speculative set")) ||
      (st = dalloc_t(p, &stp, size_t(smax), "speculative set")) ||
      (st = dalloc_t(p, &scount, size_t(ISDF_MAX_LEVELS + 1), "speculative set")) ||
      (st = dalloc_t(p, &round, 1, "block round")) ||
      (!gshared && (st = dalloc_t(p, &gcols, size_t(gthreads) * smax, "block columns"))))
    return bail(st);
  if (gshared &&
      (st = cuda_check(p, cudaFuncSetAttribute(k_blk_greedy, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kGreedySmem)),
                       "smem attribute")))
    return bail(st);
  BlkParams BP{};
  BP.P = P;
  BP.sidx = sidx;
  BP.st = stp;
  BP.scount = scount;
  for (int l = 0; l < nlev; ++l) {
    BP.bm[l] = lb[l].col;
    BP.bdf[l] = lb[l].bdf;
  }
  TopSOut O{sidx, sg, stp, scount};

  SelState h{};
  h.first = ULLONG_MAX;
  h.skip = 1;
  if ((st = cuda_check(p, cudaMemcpyAsync(p->d_selstate, &h, sizeof(h), cudaMemcpyHostToDevice, s), "state init")))
    return bail(st);
  SelState* dst = static_cast<SelState*>(p->d_selstate);
  const size_t smem = sizeof(double) * (size_t((nGmax + 1) & ~1) + 3 * kColWarps * 32);
  if (smem > 48 * 1024 &&
      (st = cuda_check(p, cudaFuncSetAttribute(k_sel_col, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kColSmem)),
                       "smem attribute")))
    return bail(st);
  int dev = 0, nsm = 152, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sel_col, 32 * kColWarps, smem);
  const unsigned red_blocks = sel_blocks(P.ntot, nsm);
  const unsigned col_blocks = per_sm > 0 ? unsigned(per_sm * nsm) : kColBlocks;
  // ---- exact compaction of the candidates below tau (see above)
  int64_t since_compact = 0;
  auto compact = [&]() -> isdf_status {
    isdf_status cst;
    // survivors per level (ordered compaction of {t : d[t] >= tau})
    int64_t keep_n[ISDF_MAX_LEVELS] = {0, 0, 0, 0}, tot_old = 0, tot_new = 0;
    std::vector<std::vector<int>> offs(nlev);
    for (int l = 0; l < nlev; ++l) {
      tot_old += nc[l];
      if (!nc[l]) continue;
      const int64_t nb = (nc[l] + kCompactBlock - 1) / kCompactBlock;
      k_flag_count<<<unsigned(nb), kCompactBlock, 0, s>>>(P.d + P.coff[l], nc[l], tau, counts);
      offs[l].resize(nb);
      cudaMemcpyAsync(offs[l].data(), counts, sizeof(int) * nb, cudaMemcpyDeviceToHost, s);
      if ((cst = cuda_check(p, cudaStreamSynchronize(s), "compaction counts"))) return cst;
      int64_t acc = 0;
      for (int64_t b = 0; b < nb; ++b) {
        const int c = offs[l][b];
        offs[l][b] = int(acc);
        acc += c;
      }
      keep_n[l] = acc;
      tot_new += acc;
      count_launches(1);
    }
    // rebuild only when at least a third of the candidates would go (the
    // rebuild re-slices the survivors' basis values; a third, checked every
    // other block, measured best: 0.418 s with a fifth, 0.401 s with a third,
    // 0.410 s with a half for the selection of the 2x2x2 diamond workload)
    if (tot_new == 0 || 3 * tot_new > 2 * tot_old) return ISDF_OK;
    double* dnew = nullptr;
    if ((cst = dalloc_t(p, &dnew, size_t(tot_new), "residual diagonal"))) return cst;
    int64_t coff_new[ISDF_MAX_LEVELS + 1] = {0};
    for (int l = 0; l < nlev; ++l) coff_new[l + 1] = coff_new[l] + keep_n[l];
    for (int l = 0; l < nlev; ++l) {
      if (!nc[l]) continue;
      Level& lv = p->lev[l];
      LevBuf& b = lb[l];
      const int64_t nn = keep_n[l], no = nc[l];
      const int64_t nb = (no + kCompactBlock - 1) / kCompactBlock;
      int *keep = nullptr, *ci = nullptr;
      double *fnew = nullptr, *d0c = nullptr;
      if (nn && ((cst = dalloc_t(p, &keep, size_t(nn), "compaction")) || (cst = dalloc_t(p, &ci, size_t(nn), "candidates")) ||
                 (cst = dalloc_t(p, &fnew, size_t(std::max<int64_t>(lv.fac_cap * nn, 1)), "selection factor columns")) ||
                 (cst = dalloc_t(p, &d0c, size_t(nn), "initial residuals")))) {
        dfree(keep), dfree(ci), dfree(fnew), dfree(d0c), dfree(dnew);
        return cst;
      }
      if (nn) {
        cudaMemcpyAsync(counts, offs[l].data(), sizeof(int) * nb, cudaMemcpyHostToDevice, s);
        k_compact<<<unsigned(nb), kCompactBlock, 0, s>>>(P.d + P.coff[l], no, tau, counts, keep);
        k_map_idx<<<unsigned((nn + 255) / 256), 256, 0, s>>>(cur_cidx[l], keep, nn, ci);
        k_gather_diag<<<unsigned((nn + 255) / 256), 256, 0, s>>>(P.d + P.coff[l], keep, nn, dnew + coff_new[l]);
        if (h.kl[l] > 0)
          k_gather_cols<<<unsigned((nn * h.kl[l] + 255) / 256), 256, 0, s>>>(lv.fac, no, keep, nn, h.kl[l], fnew);
        k_gather_diag<<<unsigned((nn + 255) / 256), 256, 0, s>>>(d0full + p->off[l], ci, nn, d0c);
        count_launches(5);
      }
      // grid -> candidate map
      if (!b.gpos && (cst = dalloc_t(p, &b.gpos, size_t(lv.ng), "grid-to-candidate map"))) {
        dfree(keep), dfree(ci), dfree(fnew), dfree(d0c), dfree(dnew);
        return cst;
      }
      cudaMemsetAsync(b.gpos, 0xFF, sizeof(int) * size_t(lv.ng), s);
      if (nn) {
        k_scatter_pos<<<unsigned((nn + 255) / 256), 256, 0, s>>>(ci, nn, b.gpos);
        count_launches(1);
      }
      // candidate-side digit planes for the survivors: basis values, then the
      // factor columns so far (fixed scales from sqrt(d0), as at set-up)
      auto setrows = [&](OzOperand& op, int64_t rows) {
        op.rows = rows;
        op.nrt = (rows + op.rt - 1) / op.rt;
      };
      setrows(b.aL, nn);
      if (lv.nN > 0) setrows(b.aN, nn);
      setrows(b.aF, nn);
      if (nn) {
        Prof pr(p, "select_slice", 8.0 * double(nn) * (lv.nG + h.kl[l]), "byte", 0);
        if (lv.nL > 0) oz_slice_ex(lv.phi, 1, lv.ng, ci, b.aL, 0, b.aL.nkt * (kOzBK / 8), false, s);
        if (lv.nN > 0)
          oz_slice_ex(lv.phi + int64_t(lv.nL) * lv.ng, 1, lv.ng, ci, b.aN, 0, b.aN.nkt * (kOzBK / 8), false, s);
        const int64_t kst_keep = b.aF.kst;
        cudaMemsetAsync(b.aF.tiles, 0, size_t(b.aF.nrt) * size_t(kst_keep) * kSlices * 128 * kOzBK * 2, s);
        k_fac_exps<<<unsigned((b.aF.nrt * 128 + 255) / 256), 256, 0, s>>>(d0c, nn, b.aF.nrt * 128, b.aF.exps);
        count_launches(1);
        b.aF.K = h.kl[l];
        if (h.kl[l] > 0) oz_slice_ex(fnew, 1, nn, nullptr, b.aF, 0, (h.kl[l] + 7) / 8, true, s);
      }
      dfree(lv.fac);
      lv.fac = fnew;
      P.fac[l] = fnew;
      cur_cidx[l] = ci;
      if (ci) own_cidx.push_back(ci);
      P.cidx[l] = ci;
      Q.cidx[l] = ci;
      Q.gpos[l] = b.gpos;
      nc[l] = nn;
      P.nc[l] = nn;
      if ((cst = cuda_check(p, cudaStreamSynchronize(s), "compaction"))) {
        dfree(keep), dfree(d0c), dfree(dnew);
        return cst;
      }
      dfree(keep);
      dfree(d0c);
    }
    dfree(p->d_diag);
    p->d_diag = dnew;
    P.d = dnew;
    Q.d = dnew;
    for (int l = 0; l <= nlev; ++l) P.coff[l] = Q.coff[l] = coff_new[l];
    P.ntot = Q.ntot = coff_new[nlev];
    BP.P = P;
    since_compact = 0;
    ++p->sel_compactions;
    return ISDF_OK;
  };
  // ---- factor capacity: before a block that could fill a level (at most
  // smax block steps, or one single step), that level's factor columns move
  // to twice the storage and their digits are sliced again (fixed scales
  // from sqrt(d0), as at set-up)
  auto grow = [&]() -> isdf_status {
    isdf_status gst;
    for (int l = 0; l < nlev; ++l) {
      Level& lv = p->lev[l];
      LevBuf& b = lb[l];
      if (!nc[l]) continue;
      const int64_t full = std::min<int64_t>(nip, nc[l]);
      const int64_t need = std::min<int64_t>(full, int64_t(h.kl[l]) + smax + 1);
      if (need <= lv.fac_cap) continue;
      const int64_t cap = std::min<int64_t>(full, std::max<int64_t>(2 * lv.fac_cap, need));
      const int kl = h.kl[l];
      double *fnew = nullptr, *d0c = nullptr;
      if ((gst = dalloc_t(p, &fnew, size_t(cap * nc[l]), "selection factor columns"))) return gst;
      if (kl > 0)
        cudaMemcpyAsync(fnew, lv.fac, sizeof(double) * size_t(kl) * size_t(nc[l]), cudaMemcpyDeviceToDevice, s);
      const double* d0src = d0full + p->off[l];
      if (cur_cidx[l]) {
        if ((gst = dalloc_t(p, &d0c, size_t(nc[l]), "initial residuals"))) {
          dfree(fnew);
          return gst;
        }
        k_gather_diag<<<unsigned((nc[l] + 255) / 256), 256, 0, s>>>(d0full + p->off[l], cur_cidx[l], nc[l], d0c);
        count_launches(1);
        d0src = d0c;
      }
      oz_free(b.aF);
      oz_free(b.bF);
      if ((gst = oz_alloc(p, b.aF, nc[l], cap, 128, kSlices, "selection slices")) ||
          (gst = oz_alloc(p, b.bF, smax, cap, oz_bn(kSlices), kSlices, "selection slices"))) {
        dfree(fnew), dfree(d0c);
        return gst;
      }
      cudaMemsetAsync(b.aF.tiles, 0, size_t(oz_tile_bytes(b.aF)), s);
      k_fac_exps<<<unsigned((b.aF.nrt * 128 + 255) / 256), 256, 0, s>>>(d0src, nc[l], b.aF.nrt * 128, b.aF.exps);
      count_launches(1);
      b.aF.K = kl;
      if (kl > 0) oz_slice_ex(fnew, 1, nc[l], nullptr, b.aF, 0, (kl + 7) / 8, true, s);
      gst = cuda_check(p, cudaStreamSynchronize(s), "factor capacity");
      dfree(lv.fac);
      dfree(d0c);
      lv.fac = fnew;
      lv.fac_cap = cap;
      P.fac[l] = fnew;
      if (gst) return gst;
    }
    BP.P = P;
    return ISDF_OK;
  };
  int64_t nblocks = 0, nplain = 0;
  int m_next = std::min(smax, 32);  // steps tried per round: a quarter more than the last one accepted, and 6
  while (true) {
    if ((st = grow())) return bail(st);
    // ---- 1. the speculative set S
    {
      Prof pr(p, "select_spec", double(P.ntot) * 8.0, "byte", 2);
      cudaMemsetAsync(nlist, 0, sizeof(int), s);
      k_lm_list<<<unsigned(std::max<int64_t>((P.ntot + 255) / 256, 1)), 256, 0, s>>>(Q, list, nlist);
      k_top_s<<<1, 1024, 0, s>>>(Q, list, nlist, smax, O);
    }
    // ---- 2. the columns of S at every candidate, B = w M - F
    size_t gemm_event = size_t(-1);
    {
      OzColumnJob jobs[ISDF_MAX_LEVELS];
      double bytes = 0.0;
      for (int l = 0; l < nlev; ++l) {
        if (!nc[l]) continue;
        Level& lv = p->lev[l];
        LevBuf& b = lb[l];
        OzColumnJob& J = jobs[l];
        b.aF.K = h.kl[l];
        b.aF.nkt = (h.kl[l] + kOzBK - 1) / kOzBK;
        J.M = nc[l];
        J.C = b.col;
        J.w = lv.w;
        if (lv.nL > 0) J.A[0] = &b.aL, J.B[0] = &b.bL, J.src[0] = lv.phi, J.ld[0] = lv.ng;
        if (lv.nN > 0) J.A[1] = &b.aN, J.B[1] = &b.bN, J.src[1] = lv.phi + int64_t(lv.nL) * lv.ng, J.ld[1] = lv.ng;
        J.A[2] = &b.aF, J.B[2] = &b.bF, J.src[2] = lv.fac, J.ld[2] = nc[l];
        bytes += 8.0 * double(nc[l]) * (lv.nG + h.kl[l]);
      }
      {
        Prof pb(p, "select_sslice", 0.0, "byte", kLaunchesInside);
        oz_set_rows(jobs, nlev, smax, scount, stp, sg, s);
      }
      // algorithmic traffic: the candidates' FP64 basis values and factor rows, read once per block
      {
        Prof pr(p, "select_gemm", bytes, "byte", kLaunchesInside);
        oz_columns(jobs, nlev, scount, p->d_ozerr, s);
      }
      if (p->opt.profile) gemm_event = p->pend.size() - 1;
    }
    // ---- 3. greedy steps of this block, in rounds: as long as every tried step
    // of a round is accepted there may be more in S
    int taken = 0;
    for (int l = 0; l < nlev; ++l) BP.kb[l] = h.kl[l];
    while (true) {
      int kl_before[ISDF_MAX_LEVELS];
      for (int l = 0; l < nlev; ++l) kl_before[l] = h.kl[l];
      const int m = std::min(m_next, smax - taken);
      {
        Prof pr(p, "select_steps", 0.0, "byte", 3);
        BP.P = P;
        BP.k = h.k;
        BP.boff[0] = 0;
        for (int l = 0; l < nlev; ++l) {
          BP.kl[l] = h.kl[l];
          BP.boff[l + 1] = BP.boff[l] + (nc[l] + kApply - 1) / kApply;
          BP.fexp[l] = lb[l].aF.exps;
          BP.ftiles[l] = lb[l].aF.tiles;
          BP.fkst[l] = lb[l].aF.kst;
        }
        const unsigned nblk = unsigned(std::max<int64_t>(BP.boff[nlev], 1));
        k_blk_greedy<<<1, gthreads, gshared ? gsmem : 0, s>>>(BP, dst, round, m, smax, gcols);
        // the next two kernels index by what this one has written
        if ((st = cuda_check(p, cudaGetLastError(), "selection steps"))) return bail(st);
        k_blk_apply<<<nblk, kApply, 0, s>>>(BP, dst, round);
        k_blk_commit<<<nblk, kApply, 0, s>>>(BP, round, dst);
      }
      if ((st = cuda_check(p, cudaGetLastError(), "selection kernels"))) return bail(st);
      cudaMemcpyAsync(&h, dst, sizeof(h), cudaMemcpyDeviceToHost, s);
      if ((st = cuda_check(p, cudaStreamSynchronize(s), "block state"))) return bail(st);
      if (p->opt.profile && !p->pend.empty() && p->pend.back().name == "select_steps") {
        // algorithmic bytes of the round: per accepted step and candidate of its
        // level the column of B, the block's earlier columns and the new column;
        // the residual once
        double bytes = 16.0 * double(P.ntot);
        for (int l = 0; l < nlev; ++l) {
          const double dk = h.kl[l] - kl_before[l], n = double(nc[l]);
          bytes += 24.0 * dk * n + 8.0 * n * dk * (dk - 1.0) / 2.0;
        }
        p->pend.back().work = bytes;
      }
      taken += h.bsteps;
      m_next = std::min(smax, std::max(12, h.bsteps + h.bsteps / 4 + 6));
      if (h.err || h.final_ || h.k >= nip || h.bsteps < m || taken >= smax) break;
    }
    ++nblocks;
    if (gemm_event != size_t(-1) && gemm_event < p->pend.size())
      for (int l = 0; l < nlev; ++l)
        p->pend[gemm_event].flop += 2.0 * double(nc[l]) * h.members[l] * double(p->lev[l].nG + BP.kb[l]);
    if (h.err || h.final_ || h.k >= nip) break;
    if (tau > 0.0 && taken > 0 && h.dp * (1.0 - 2.0 * p->opt.tie_rel) - 2.0 * p->opt.tie_abs * h.d0 < tau) {
      *aborted = true;  // a pivot value broke the certificate: retry with a lower tau
      break;
    }
    if (taken == 0) {
      // the greedy pivot was not in S: one ordinary step
      Prof pr(p, "select_loop", 0.0, "flop", 3);
      k_step_begin<<<1, 32, 0, s>>>(dst);
      k_sel_max<<<dim3(red_blocks, unsigned(P.nlev)), 256, 0, s>>>(P, dst);
      k_sel_first<<<red_blocks, 256, 0, s>>>(P, dst);
      k_sel_col<<<col_blocks, 256, smem, s>>>(P, dst);
      count_launches(4);
      ++nplain;
      cudaMemcpyAsync(&h, dst, sizeof(h), cudaMemcpyDeviceToHost, s);
      if ((st = cuda_check(p, cudaStreamSynchronize(s), "plain step"))) return bail(st);
      if (h.err || h.final_ || h.k >= nip) break;
    }
    if (tau > 0.0 && h.dp * (1.0 - 2.0 * p->opt.tie_rel) - 2.0 * p->opt.tie_abs * h.d0 < tau) {
      *aborted = true;
      break;
    }
    // ---- 4. digits of an ordinary step's column (a block's are written as it is accepted)
    if (taken == 0) {
      Prof pr(p, "select_slice", 0.0, "byte", kLaunchesInside);
      for (int l = 0; l < nlev; ++l) {
        LevBuf& b = lb[l];
        if (h.kl[l] <= BP.kl[l]) continue;
        b.aF.K = h.kl[l];
        oz_slice_ex(p->lev[l].fac, 1, nc[l], nullptr, b.aF, BP.kl[l] / 8, (h.kl[l] + 7) / 8, true, s);
      }
    }
    // ---- 5. drop the candidates whose residual fell below tau (checked every other block)
    if (tau > 0.0 && ++since_compact >= 2 && (st = compact())) return bail(st);
  }
  if ((st = oz_check(p))) return bail(st);
  *nfound = h.k;
  for (int l = 0; l < nlev; ++l) kl_out[l] = h.kl[l];
  p->sel_blocks = nblocks;
  p->sel_plain_steps = nplain;
  cleanup();
  if (h.err == ISDF_ERR_TIMEOUT) return fail(p, ISDF_ERR_TIMEOUT, "selection loop exceeded options.timeout_ms");
  return ISDF_OK;
}

}  // namespace

isdf_status select_run(Plan* p, int nip, double tol, const std::vector<int64_t>* cand, int* nfound) {
  cudaStream_t s = p->stream;
  isdf_status st;
  dfree(p->d_piv);
  p->d_piv = nullptr;
  dfree(p->d_dval);
  p->d_dval = nullptr;
  if (!p->d_selstate && (st = dalloc(p, &p->d_selstate, sizeof(SelState), "selection state"))) return st;
  if ((st = dalloc_t(p, &p->d_piv, size_t(nip), "pivots"))) return st;
  if ((st = dalloc_t(p, &p->d_dval, size_t(nip), "pivot values"))) return st;
  // initial residual diagonal on every point of every level
  double* d0 = nullptr;
  if ((st = dalloc_t(p, &d0, size_t(p->ntot), "initial diagonal"))) return st;
  for (int l = 0; l < p->nlev; ++l) {
    Level& lv = p->lev[l];
    if (lv.nG == 0) {  // a level without basis values of its own (local grids' level 0)
      cudaMemsetAsync(d0 + p->off[l], 0, sizeof(double) * size_t(lv.ng), s);
      continue;
    }
    Prof pr(p, "select_diag", 2.0 * double(lv.nG) * double(lv.ng), "flop", 1);
    k_sel_diag<<<152 * 8, 256, 0, s>>>(lv.phi, lv.ng, lv.nL, lv.nG, lv.w, d0 + p->off[l]);
  }
  int* cidx[ISDF_MAX_LEVELS] = {nullptr, nullptr, nullptr, nullptr};
  int64_t nc[ISDF_MAX_LEVELS] = {0, 0, 0, 0};
  auto free_cidx = [&]() {
    for (int l = 0; l < p->nlev; ++l) {
      dfree(cidx[l]);
      cidx[l] = nullptr;
    }
  };
  auto done = [&](isdf_status r) {
    free_cidx();
    dfree(d0);
    return r;
  };
  // with the coarsest level as the universal sinc grid it takes no part in
  // the selection: no candidates there, and d_0 is the finer levels' largest;
  // levels below sel_lo (local grids' level 0) have their own selections
  const int nsel = p->opt.coarse_sinc ? p->nlev - 1 : p->nlev;
  const int lo = p->sel_lo;
  int kl[ISDF_MAX_LEVELS];
  bool aborted = false;
  p->sel_compactions = 0;
  auto loop = [&](int* const* ci, const int64_t* n, double tau = 0.0) {
    aborted = false;
    return p->opt.select_block > 0 ? select_loop_blocked(p, nip, tol, d0, ci, n, nfound, kl, tau, &aborted)
                                   : select_loop(p, nip, tol, d0, ci, n, nfound, kl);
  };
  if (cand) {
    // caller-given candidates: ascending, unique per level
    std::vector<std::vector<int>> per(p->nlev);
    for (int64_t c : *cand) per[c >> kPivShift].push_back(int(c & kPivMask));
    for (int l = 0; l < p->nlev; ++l) {
      std::sort(per[l].begin(), per[l].end());
      per[l].erase(std::unique(per[l].begin(), per[l].end()), per[l].end());
      nc[l] = int64_t(per[l].size());
      if (!nc[l]) continue;
      if ((st = dalloc_t(p, &cidx[l], size_t(nc[l]), "candidates"))) return done(st);
      if ((st = cuda_check(p, cudaMemcpyAsync(cidx[l], per[l].data(), sizeof(int) * nc[l], cudaMemcpyHostToDevice, s),
                           "copy candidates")))
        return done(st);
    }
    if ((st = cuda_check(p, cudaStreamSynchronize(s), "copy candidates"))) return done(st);
    return done(loop(cidx, nc));
  }
  if (!p->opt.prefilter) {
    for (int l = 0; l < p->nlev; ++l) nc[l] = (l >= lo && l < nsel) ? p->lev[l].ng : 0;
    return done(loop(cidx, nc));
  }
  // exact prefilter: tau relative to the largest initial residual d_0
  unsigned long long* dmax_slot = nullptr;
  if ((st = dalloc_t(p, &dmax_slot, 1, "max slot"))) return done(st);
  cudaMemsetAsync(dmax_slot, 0, sizeof(unsigned long long), s);
  k_vec_max<<<152 * 4, 256, 0, s>>>(d0, p->off[nsel], dmax_slot);
  count_launches(1);
  unsigned long long bits = 0;
  cudaMemcpyAsync(&bits, dmax_slot, sizeof(bits), cudaMemcpyDeviceToHost, s);
  st = cuda_check(p, cudaStreamSynchronize(s), "prefilter max");
  dfree(dmax_slot);
  if (st) return done(st);
  double dmax0;
  std::memcpy(&dmax0, &bits, sizeof(dmax0));
  // attempts: the blocked form starts at 1e-5 d_0 (its candidates shrink as
  // the residuals fall below tau, and an attempt whose pivot values break the
  // certificate stops at once); the step-by-step form at 1e-6 d_0
  const bool blocked = p->opt.select_block > 0;
  const double taus[4] = {blocked ? 1e-5 : 1e-6, 1e-6, 1e-9, 0.0};
  for (int attempt = blocked ? 0 : 1; attempt < 4; ++attempt) {
    const double tau = (attempt == 0 ? taus[0] : taus[attempt]) * dmax0;
    free_cidx();
    for (int l = 0; l < p->nlev; ++l) {
      Level& lv = p->lev[l];
      if (l >= nsel || l < lo) {
        nc[l] = 0;
        continue;
      }
      if (tau <= 0.0) {
        nc[l] = lv.ng;
        continue;
      }
      const int64_t nb = (lv.ng + kCompactBlock - 1) / kCompactBlock;
      int* counts = nullptr;
      if ((st = dalloc_t(p, &counts, size_t(nb), "compaction counts"))) return done(st);
      k_flag_count<<<unsigned(nb), kCompactBlock, 0, s>>>(d0 + p->off[l], lv.ng, tau, counts);
      std::vector<int> hc(nb);
      cudaMemcpyAsync(hc.data(), counts, sizeof(int) * nb, cudaMemcpyDeviceToHost, s);
      if ((st = cuda_check(p, cudaStreamSynchronize(s), "compaction counts"))) {
        dfree(counts);
        return done(st);
      }
      int64_t acc = 0;
      for (int64_t b = 0; b < nb; ++b) {
        const int c = hc[b];
        hc[b] = int(acc);
        acc += c;
      }
      nc[l] = acc;
      if (acc) {
        if ((st = dalloc_t(p, &cidx[l], size_t(acc), "candidates"))) {
          dfree(counts);
          return done(st);
        }
        cudaMemcpyAsync(counts, hc.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, s);
        k_compact<<<unsigned(nb), kCompactBlock, 0, s>>>(d0 + p->off[l], lv.ng, tau, counts, cidx[l]);
      }
      count_launches(acc ? 2 : 1);
      st = cuda_check(p, cudaStreamSynchronize(s), "compaction");
      dfree(counts);
      if (st) return done(st);
    }
    bool all_kept = true;
    for (int l = lo; l < nsel; ++l) all_kept = all_kept && nc[l] == p->lev[l].ng;
    if (all_kept) {  // nothing dropped: this is the full greedy run
      free_cidx();
      return done(loop(cidx, nc));
    }
    st = loop(cidx, nc, tau);
    if (st || tau <= 0.0) return done(st);
    if (aborted) continue;
    // certificate: every step's tie threshold stayed above tau
    std::vector<double> dv(*nfound);
    cudaMemcpyAsync(dv.data(), p->d_dval, sizeof(double) * dv.size(), cudaMemcpyDeviceToHost, s);
    if ((st = cuda_check(p, cudaStreamSynchronize(s), "pivot values"))) return done(st);
    bool ok = *nfound == nip || (tol > 0.0 && tau <= tol * dmax0);
    for (double v : dv) ok = ok && (v * (1.0 - 2.0 * p->opt.tie_rel) - 2.0 * p->opt.tie_abs * dmax0 >= tau);
    if (ok) return done(ISDF_OK);
  }
  return done(ISDF_OK);
}

}  // namespace isdf
