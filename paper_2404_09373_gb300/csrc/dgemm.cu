// FP64 SIMT dense kernels: tiled GEMM, the fused Hadamard GEMM of the fit,
// blocked Cholesky and triangular inverse.  These are the "plain FP64" form of
// the contractions (options.precision = 0); the Cholesky and the small blocks
// of the inverse serve both precisions.
//
// The FP64 unit (2 FMA per clock and SM) bounds all of them: an SM needs 16 us
// for a 32 x 32 tile over 64 k values, while the operands of that tile are 32
// KB from L2.  So the tiles are small: no padding beyond 32, and work for every
// SM as early as possible; a larger tile would only save loads, which are free.
#include <algorithm>

#include "dfloat.cuh"
#include "internal.cuh"

namespace isdf {
namespace {

constexpr int BT = 32, BK = 32, NT = 128;  // output tile, k step, threads (2 x 4 outputs each)
constexpr int RI = 2, RJ = 4;

struct Tiles {
  double a[BK][BT + 1];
  double b[BK][BT + 1];
};

// Accumulate acc[i][j] += sum_{k in [kbeg,kend)} opA(m0+ty+16i, k) w(k) opB(k, n0+tx+8j).
template <int TA, int TB>
__device__ __forceinline__ void tile_accumulate(double (&acc)[RI][RJ], Tiles& t, const double* __restrict__ A,
                                                int64_t lda, const double* __restrict__ B, int64_t ldb,
                                                const double* __restrict__ kw, int64_t M, int64_t N, int64_t m0,
                                                int64_t n0, int64_t kbeg, int64_t kend) {
  const int tid = threadIdx.x;
  const int tx = tid % 8, ty = tid / 8;
  const int fast = tid % 32, slow = tid / 32;  // loads: 32 consecutive elements per warp
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int q = 0; q < BT; q += NT / 32) {
      const int kk = TA ? slow + q : fast, mm = TA ? fast : slow + q;
      const int64_t gk = k0 + kk, gm = m0 + mm;
      double v = 0.0;
      if (gk < kend && gm < M) {
        v = TA ? A[gk * lda + gm] : A[gm * lda + gk];
        if (kw) v *= kw[gk];
      }
      t.a[kk][mm] = v;
    }
#pragma unroll
    for (int q = 0; q < BT; q += NT / 32) {
      const int kk = TB ? fast : slow + q, nn = TB ? slow + q : fast;
      const int64_t gk = k0 + kk, gn = n0 + nn;
      double v = 0.0;
      if (gk < kend && gn < N) v = TB ? B[gn * ldb + gk] : B[gk * ldb + gn];
      t.b[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      double av[RI], bv[RJ];
#pragma unroll
      for (int i = 0; i < RI; ++i) av[i] = t.a[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < RJ; ++j) bv[j] = t.b[kk][tx + 8 * j];
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
}

// visit(m, n, acc value) for this thread's outputs inside M x N
template <class F>
__device__ __forceinline__ void tile_visit(const double (&acc)[RI][RJ], int64_t M, int64_t N, int64_t m0, int64_t n0,
                                           F visit) {
  const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    const int64_t m = m0 + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
      const int64_t n = n0 + tx + 8 * j;
      if (n < N) visit(m, n, acc[i][j]);
    }
  }
}

// gridDim.z > 1: each z takes a share of the tile's k range and leaves its sum
// in work[z][M][N] (k_dgemm_sum adds them in order)
template <int TA, int TB>
__global__ __launch_bounds__(NT) void k_dgemm(GemmArgs g, double* __restrict__ work) {
  const int64_t m0 = int64_t(blockIdx.y) * BT, n0 = int64_t(blockIdx.x) * BT;
  if (g.sym && n0 > m0 + BT - 1) return;
  __shared__ Tiles t;
  double acc[RI][RJ] = {};
  int64_t kbeg = 0, kend = g.K;
  if (g.tri == 1) kend = (m0 + BT < g.K) ? m0 + BT : g.K;
  if (g.tri == 2) kbeg = m0;
  if (gridDim.z > 1) {
    const int64_t steps = (kend - kbeg + BK - 1) / BK, per = (steps + gridDim.z - 1) / gridDim.z;
    kbeg += per * blockIdx.z * BK;
    kend = kbeg + per * BK < kend ? kbeg + per * BK : kend;
  }
  tile_accumulate<TA, TB>(acc, t, g.A, g.lda, g.B, g.ldb, g.kw, g.M, g.N, m0, n0, kbeg, kend);
  if (work) {
    double* w = work + int64_t(blockIdx.z) * g.M * g.N;
    tile_visit(acc, g.M, g.N, m0, n0, [&](int64_t m, int64_t n, double v) { w[m * g.N + n] = v; });
    return;
  }
  tile_visit(acc, g.M, g.N, m0, n0, [&](int64_t m, int64_t n, double x) {
    double* c = g.C + m * g.ldc + n;
    const double v = g.alpha * x;
    *c = (g.beta == 0.0) ? v : fma(g.beta, *c, v);
  });
}

__global__ void k_dgemm_sum(GemmArgs g, const double* __restrict__ work, int splits) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= g.M * g.N) return;
  const int64_t m = e / g.N, n = e % g.N;
  if (g.sym && n / BT > m / BT) return;
  double s = 0.0;
  for (int z = 0; z < splits; ++z) s += work[int64_t(z) * g.M * g.N + e];
  double* c = g.C + m * g.ldc + n;
  const double v = g.alpha * s;
  *c = (g.beta == 0.0) ? v : fma(g.beta, *c, v);
}

// (ZC^T)^T[j][g] = aL (aL + 2 aN), aL = sum_{r<nL} phiP[r][j] phi[r][g],
// aN = sum_{nL<=r<nG} phiP[r][j] phi[r][g]   (M_l[:, P], Eq. 2 / Eq. 3)
__global__ __launch_bounds__(NT) void k_zc(int64_t k, int64_t ng, int nL, int nG, const double* __restrict__ phiP,
                                           const double* __restrict__ phi, double* __restrict__ out) {
  const int64_t m0 = int64_t(blockIdx.y) * BT, n0 = int64_t(blockIdx.x) * BT;
  __shared__ Tiles t;
  double aL[RI][RJ] = {}, aN[RI][RJ] = {};
  tile_accumulate<1, 0>(aL, t, phiP, k, phi, ng, nullptr, k, ng, m0, n0, 0, nL);
  tile_accumulate<1, 0>(aN, t, phiP, k, phi, ng, nullptr, k, ng, m0, n0, nL, nG);
#pragma unroll
  for (int i = 0; i < RI; ++i)
#pragma unroll
    for (int j = 0; j < RJ; ++j) aL[i][j] = aL[i][j] * (aL[i][j] + 2.0 * aN[i][j]);
  tile_visit(aL, k, ng, m0, n0, [&](int64_t m, int64_t n, double v) { out[m * ng + n] = v; });
}

// ---- Cholesky (right-looking, 64-column blocks) and inverse of the factor ----
//
// All levels go through the same launches (blockIdx.y or .z = level), and a
// block column costs two of them:
//   k_chol_panel   X = A R_kk^-T as a product with the inverted diagonal block
//   k_chol_update  trailing tiles -= X X^T; the CTA that finishes the last tile
//                  of the next diagonal block factors and inverts that block at
//                  once, under the rest of the update (an atomic count, no waiting)
// so the serial part, the 64 dependent columns, is hidden wherever the update is
// longer.  The inverted diagonal blocks are those of R^-1, where
// dtrtri_lower starts.
//
// A product with the inverted block leaves an error of eps cond(R_kk) |A| in a
// block column where a substitution leaves eps |A|.  Residual |A - R R^T| / |A|
// emulated for CC^T of one cell at 6 points a function (cond(CC^T) up to 1e6, of
// the 64 x 64 blocks up to 50 in selection order, 700 in grid order): 1.2 to
// 2.8e-16 against 1.0 to 2.3e-16 by substitution.  64 neighbouring grid points
// first (block 7e5, CC^T 1e14): 1.2e-15 against 1.1e-16.
constexpr int CB = 64;

struct CholLevel {
  double* A;   // n x n, lower triangle factored in place
  double* Li;  // n x n, R^-1
  double* T;   // scratch of the inverse
  int n;
  int* err;    // smallest column whose pivot was not positive
  int* count;  // per block column: finished tiles of its diagonal block
};
struct CholLevels {
  CholLevel l[ISDF_MAX_LEVELS];
};

struct DiagSmem {
  double s[CB][CB + 1];
  double v[CB][CB + 1];
  double t[CB / 2][CB / 2 + 1];
  double r[CB];  // reciprocals of the diagonal
};

// Factor the b x b diagonal block at kb and invert the factor (all NT threads).
__device__ void chol_diag(const CholLevel& P, int kb, DiagSmem& S) {
  const int tid = threadIdx.x, n = P.n, b = n - kb < CB ? n - kb : CB;
  for (int e = tid; e < CB * CB; e += NT) {
    const int i = e / CB, c = e % CB;
    // written by other CTAs of this launch: read past L1
    S.s[i][c] = (i < b && c <= i) ? __ldcg(P.A + int64_t(kb + i) * n + kb + c) : (i == c ? 1.0 : 0.0);
    S.v[i][c] = 0.0;
  }
  __syncthreads();
  for (int j = 0; j < b; ++j) {
    if (tid < 32) {
      double d = S.s[j][j];
      if (!(d > 0.0) || !isfinite(d)) {
        if (tid == 0) atomicMin(P.err, kb + j);
        d = 1.0;
      }
      const double r = root64(d).r;
      // the column below the diagonal, two rows a lane (rows at or above j stay)
      const int i0 = tid, i1 = tid + 32;
      const double x0 = S.s[i0][j], x1 = S.s[i1][j];
      __syncwarp();  // the diagonal is read by every lane before it is replaced
      if (i0 > j) S.s[i0][j] = x0 * r;
      if (i1 > j) S.s[i1][j] = x1 * r;
      if (tid == 0) {
        S.r[j] = r;
        S.s[j][j] = d;  // no later column reads it: the roots are taken together below
      }
    }
    __syncthreads();
    // two threads per row; columns c in (j, i]
    const int i = tid >> 1;
    if (i > j && i < b) {
      const double x = S.s[i][j];
      for (int c = j + 1 + (tid & 1); c <= i; c += 2) S.s[i][c] = fma(-x, S.s[c][j], S.s[i][c]);
    }
    __syncthreads();
  }
  // inverse by doubling: [A 0; C B]^-1 = [A^-1 0; -B^-1 C A^-1  B^-1]
  for (int i = tid; i < CB; i += NT) {
    if (i < b) S.s[i][i] = root64(S.s[i][i]).s;
    S.v[i][i] = i < b ? S.r[i] : 1.0;
  }
  __syncthreads();
  for (int h = 1; h < CB; h *= 2) {
    const int per = h * h, tot = (CB / (2 * h)) * per;  // <= 32 * 64 / 2
    // T = C A^-1, element (i, j) of pair q at t[flat]
    double* t = &S.t[0][0];
    for (int e = tid; e < tot; e += NT) {
      const int q = e / per, i = e % h, j = (e % per) / h, r0 = 2 * h * q;
      double x = 0.0;
      for (int k = j; k < h; ++k) x = fma(S.s[r0 + h + i][r0 + k], S.v[r0 + k][r0 + j], x);
      t[q * per + j * h + i] = x;
    }
    __syncthreads();
    for (int e = tid; e < tot; e += NT) {
      const int q = e / per, i = e % h, j = (e % per) / h, r0 = 2 * h * q;
      double x = 0.0;
      for (int k = 0; k <= i; ++k) x = fma(S.v[r0 + h + i][r0 + h + k], t[q * per + j * h + k], x);
      S.v[r0 + h + i][r0 + j] = -x;
    }
    __syncthreads();
  }
  for (int e = tid; e < b * b; e += NT) {
    const int i = e / b, c = e % b;
    P.A[int64_t(kb + i) * n + kb + c] = (c <= i) ? S.s[i][c] : 0.0;
    P.Li[int64_t(kb + i) * n + kb + c] = (c <= i) ? S.v[i][c] : 0.0;
  }
}

__global__ __launch_bounds__(NT) void k_chol_first(CholLevels L) {
  extern __shared__ __align__(16) unsigned char sm_chol[];
  const CholLevel& P = L.l[blockIdx.x];
  if (P.n > 0) chol_diag(P, 0, *reinterpret_cast<DiagSmem*>(sm_chol));
}

// Rows [kb + 64, n) of block column kb: X = A R_kk^-T, 8 rows per CTA, in place.
constexpr int kPanelRows = 8;
__global__ __launch_bounds__(NT) void k_chol_panel(CholLevels L, int kb) {
  const CholLevel& P = L.l[blockIdx.y];
  const int n = P.n, r0 = kb + CB + int(blockIdx.x) * kPanelRows;
  if (r0 >= n) return;  // the block column has rows below it: kb + 64 < n, a full diagonal block
  __shared__ double a[kPanelRows][CB + 1];
  __shared__ double v[CB][CB + 1];
  const int tid = threadIdx.x;
  for (int e = tid; e < CB * CB; e += NT) v[e / CB][e % CB] = P.Li[int64_t(kb + e / CB) * n + kb + e % CB];
  for (int e = tid; e < kPanelRows * CB; e += NT) {
    const int i = e / CB;
    a[i][e % CB] = r0 + i < n ? P.A[int64_t(r0 + i) * n + kb + e % CB] : 0.0;
  }
  __syncthreads();
  // thread: rows i = tid / 32 + 4 q, columns c = lane and 63 - lane (equal work)
  const int lane = tid % 32;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int c = half ? CB - 1 - lane : lane;
    double x[kPanelRows / 4] = {};
    for (int k = 0; k <= c; ++k) {
      const double w = v[c][k];
#pragma unroll
      for (int q = 0; q < kPanelRows / 4; ++q) x[q] = fma(a[tid / 32 + 4 * q][k], w, x[q]);
    }
#pragma unroll
    for (int q = 0; q < kPanelRows / 4; ++q) {
      const int i = tid / 32 + 4 * q;
      if (r0 + i < n) P.A[int64_t(r0 + i) * n + kb + c] = x[q];
    }
  }
}

// Trailing tiles (lower triangle, 32 x 32, row by row from the next diagonal
// block) -= X X^T; then the next diagonal block, by the CTA that completes it.
__global__ __launch_bounds__(NT) void k_chol_update(CholLevels L, int kb) {
  extern __shared__ __align__(16) unsigned char sm_chol[];
  __shared__ int last;
  const CholLevel& P = L.l[blockIdx.y];
  const int n = P.n, base = kb + CB;
  const int nt = base < n ? (n - base + BT - 1) / BT : 0;  // tile rows
  const int tile = int(blockIdx.x);
  if (tile >= nt * (nt + 1) / 2) return;
  int i = int((sqrtf(8.0f * float(tile) + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > tile) --i;
  while ((i + 1) * (i + 2) / 2 <= tile) ++i;
  const int j = tile - i * (i + 1) / 2;
  Tiles& t = *reinterpret_cast<Tiles*>(sm_chol);
  double acc[RI][RJ] = {};
  const double* X = P.A + kb;
  tile_accumulate<0, 1>(acc, t, X, n, X, n, nullptr, n, n, base + BT * i, base + BT * j, 0, CB);
  tile_visit(acc, n, n, base + BT * i, base + BT * j, [&](int64_t m, int64_t c, double v) {
    double* x = P.A + m * n + c;
    *x -= v;
  });
  if (i >= CB / BT) return;  // not a tile of the next diagonal block
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int need = nt > 1 ? 3 : 1;
    last = atomicAdd(P.count + base / CB, 1) == need - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  chol_diag(P, base, *reinterpret_cast<DiagSmem*>(sm_chol));
}

// Doubling step of the inverse for half size h: node q covers rows [2hq, 2hq +
// h + n2) with both halves inverted; phase 0: T = C A^-1, phase 1: -B^-1 T.
__global__ __launch_bounds__(NT) void k_trtri_step(CholLevels L, int h, int phase) {
  const CholLevel& P = L.l[blockIdx.z];
  const int n = P.n, r0 = 2 * h * int(blockIdx.y);
  const int n2 = n - r0 - h < h ? n - r0 - h : h;
  const int tn = h / BT, m0 = (int(blockIdx.x) / tn) * BT, n0 = (int(blockIdx.x) % tn) * BT;
  if (n2 <= 0 || m0 >= n2) return;
  __shared__ Tiles t;
  double acc[RI][RJ] = {};
  double* T = P.T + int64_t(blockIdx.y) * h * h;
  const double* Lh = P.Li + int64_t(r0) * n + r0;
  if (phase == 0) {
    const double* C = P.A + int64_t(r0 + h) * n + r0;
    tile_accumulate<0, 0>(acc, t, C, n, Lh, n, nullptr, n2, h, m0, n0, n0, h);  // A^-1 lower: k >= n0
    tile_visit(acc, n2, h, m0, n0, [&](int64_t m, int64_t c, double v) { T[m * h + c] = v; });
  } else {
    const double* Bi = P.Li + int64_t(r0 + h) * n + r0 + h;
    const int ke = m0 + BT < n2 ? m0 + BT : n2;  // B^-1 lower: k <= m
    tile_accumulate<0, 0>(acc, t, Bi, n, T, h, nullptr, n2, h, m0, n0, 0, ke);
    double* out = P.Li + int64_t(r0 + h) * n + r0;
    tile_visit(acc, n2, h, m0, n0, [&](int64_t m, int64_t c, double v) { out[m * n + c] = -v; });
  }
}

}  // namespace

void dgemm(const GemmArgs& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return;
  const int64_t tm = (g.M + BT - 1) / BT, tn = (g.N + BT - 1) / BT;
  // Few tiles over a long k (the V blocks and exchange projections of a small
  // cell) leave most SMs idle: share the k range over enough CTAs for about four
  // per SM, at least 128 k values each.  The Coulomb block of a cell's 24^3 grid (about
  // 150 x 150 x 14976) has 25 tiles: 0.61 ms as 1025 CTAs.
  const int64_t tiles = g.sym ? tm * (tm + 1) / 2 : tm * tn;
  const int64_t splits = std::max<int64_t>(1, std::min<int64_t>({(608 + tiles - 1) / tiles, g.K / 128, 64}));
  double* work = nullptr;
  dim3 grid{unsigned(tn), unsigned(tm), 1u};
  if (tiles < 304 && splits > 1) {
    if (cudaMallocAsync(reinterpret_cast<void**>(&work), sizeof(double) * size_t(splits * g.M * g.N), s) == cudaSuccess) {
      grid.z = unsigned(splits);
    } else {
      cudaGetLastError();
      work = nullptr;
    }
  }
  if (g.ta == 0 && g.tb == 0) k_dgemm<0, 0><<<grid, NT, 0, s>>>(g, work);
  if (g.ta == 1 && g.tb == 0) k_dgemm<1, 0><<<grid, NT, 0, s>>>(g, work);
  if (g.ta == 0 && g.tb == 1) k_dgemm<0, 1><<<grid, NT, 0, s>>>(g, work);
  if (g.ta == 1 && g.tb == 1) k_dgemm<1, 1><<<grid, NT, 0, s>>>(g, work);
  count_launches(1);
  if (work) {
    k_dgemm_sum<<<unsigned((g.M * g.N + 255) / 256), 256, 0, s>>>(g, work, int(splits));
    count_launches(1);
    cudaFreeAsync(work, s);
  }
}

void zc_gemm(int64_t k, int64_t ng, int nL, int nG, const double* phiP, const double* phi, double* out,
             cudaStream_t s) {
  if (k <= 0 || ng <= 0) return;
  dim3 grid(unsigned((ng + BT - 1) / BT), unsigned((k + BT - 1) / BT));
  k_zc<<<grid, NT, 0, s>>>(k, ng, nL, nG, phiP, phi, out);
}

namespace {

// C (M x N, ldc) = alpha A B, A row-major (M x K, lda), B row-major (K x N,
// ldb), as an 8-digit tensor-core product; false if its buffers could not be
// allocated (the caller then takes the FP64 product)
bool tc_product(Plan* p, const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc, int64_t M,
                int64_t N, int64_t K, double alpha, cudaStream_t s) {
  OzOperand a, b;
  const bool ok = oz_alloc(p, a, M, K, 128, 8, "triangular inverse slices") == ISDF_OK &&
                  oz_alloc(p, b, N, K, oz_bn(8), 8, "triangular inverse slices") == ISDF_OK;
  if (ok) {
    oz_slice(A, lda, 1, nullptr, 1.0, a, s);
    oz_slice(B, 1, ldb, nullptr, 1.0, b, s);  // row j of the B operand: column j of B
    oz_gemm(a, b, C, ldc, 0, alpha, 0, 0, 1, nullptr, p->d_ozerr, s);
  }
  oz_free(a);
  oz_free(b);
  return ok;
}

constexpr int64_t kTcMin = 256;  // products with halves at least this large go to the tensor cores

CholLevels pack(const FactorJob* jobs, int count, int* counts, int per) {
  CholLevels L{};
  for (int i = 0; i < count; ++i)
    L.l[i] = {jobs[i].A, jobs[i].Li, jobs[i].scratch, jobs[i].n, jobs[i].err, counts ? counts + i * per : nullptr};
  return L;
}

int max_n(const FactorJob* jobs, int count) {
  int n = 0;
  for (int i = 0; i < count; ++i) n = std::max(n, jobs[i].n);
  return n;
}

}  // namespace

isdf_status dpotrf_lower(Plan* p, const FactorJob* jobs, int count, cudaStream_t s) {
  const int n = max_n(jobs, count);
  if (n <= 0) return ISDF_OK;
  const int per = (n + CB - 1) / CB + 1;
  int* counts = nullptr;
  isdf_status st = dalloc_t(p, &counts, size_t(per) * ISDF_MAX_LEVELS, "Cholesky counters");
  if (st) return st;
  cudaMemsetAsync(counts, 0, sizeof(int) * size_t(per) * ISDF_MAX_LEVELS, s);
  for (int i = 0; i < count; ++i)
    if (jobs[i].n > 0) cudaMemsetAsync(jobs[i].Li, 0, sizeof(double) * size_t(jobs[i].n) * jobs[i].n, s);
  const CholLevels L = pack(jobs, count, counts, per);
  constexpr int smem = int(sizeof(DiagSmem) > sizeof(Tiles) ? sizeof(DiagSmem) : sizeof(Tiles));
  cudaFuncSetAttribute(k_chol_first, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_chol_update, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  k_chol_first<<<unsigned(count), NT, smem, s>>>(L);
  count_launches(1);
  for (int kb = 0; kb + CB < n; kb += CB) {
    const int rows = n - kb - CB, nt = (rows + BT - 1) / BT;
    k_chol_panel<<<dim3(unsigned((rows + kPanelRows - 1) / kPanelRows), unsigned(count)), NT, 0, s>>>(L, kb);
    k_chol_update<<<dim3(unsigned(nt * (nt + 1) / 2), unsigned(count)), NT, smem, s>>>(L, kb);
    count_launches(2);
  }
  dfree(counts);
  return cuda_check(p, cudaGetLastError(), "Cholesky kernels");
}

void dtrtri_lower(Plan* p, const FactorJob* jobs, int count, bool tensor, cudaStream_t s) {
  const int n = max_n(jobs, count);
  const CholLevels L = pack(jobs, count, nullptr, 0);
  for (int h = CB; h < n; h *= 2) {
    if (tensor && h >= kTcMin)
      for (int i = 0; i < count; ++i) {
        const FactorJob& J = jobs[i];
        for (int r0 = 0; r0 + h < J.n; r0 += 2 * h) {
          const int64_t ld = J.n, n2 = std::min(h, J.n - r0 - h);
          const double* C = J.A + (r0 + h) * ld + r0;
          double* out = J.Li + (r0 + h) * ld + r0;
          if (n2 >= kTcMin && tc_product(p, C, ld, J.Li + r0 * ld + r0, ld, J.scratch, h, n2, h, h, 1.0, s) &&
              tc_product(p, J.Li + (r0 + h) * ld + r0 + h, ld, J.scratch, h, out, ld, n2, h, n2, -1.0, s))
            continue;
          GemmArgs g;  // T = C A^-1
          g.M = n2, g.N = h, g.K = h;
          g.A = C, g.lda = ld, g.B = J.Li + r0 * ld + r0, g.ldb = ld, g.C = J.scratch, g.ldc = h;
          dgemm(g, s);
          GemmArgs f;  // -B^-1 T (B^-1 lower triangular: opA(m, k) nonzero for k <= m)
          f.M = n2, f.N = h, f.K = n2, f.alpha = -1.0;
          f.A = J.Li + (r0 + h) * ld + r0 + h, f.lda = ld, f.B = J.scratch, f.ldb = h, f.C = out, f.ldc = ld, f.tri = 1;
          dgemm(f, s);
        }
      }
    else {
      const dim3 grid(unsigned((h / BT) * (h / BT)), unsigned((n - h + 2 * h - 1) / (2 * h)), unsigned(count));
      k_trtri_step<<<grid, NT, 0, s>>>(L, h, 0);
      k_trtri_step<<<grid, NT, 0, s>>>(L, h, 1);
      count_launches(2);
    }
  }
}

}  // namespace isdf
