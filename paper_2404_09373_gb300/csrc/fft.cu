// Batched 3-D real-to-half-complex DFT in double-float arithmetic: the half
// spectra S(q) = sum_r f(r) exp(-2 pi i q.r / n) (unnormalised, the layout of
// a D2Z transform: [qz][qy][qx], qx in [0, nx/2]) that the Coulomb integrals
// of Section II, Eq. 1 are built from.
//
// Every value is a pair of FP32 numbers (hi, lo) with hi + lo the represented
// number (about 48 significant bits); sums use an error-free two-sum and
// products an FMA-based two-product, so the transform runs on the FP32 pipes
// (tens of times the FP64 rate on this GPU) with an error of a few 2^-48 per
// stage relative to the vector's magnitude.
//
// One pass per axis, every line of n = R1 R2 values in two register transforms
// with one exchange through shared memory:
//   R2 threads a line: R1 values R2 apart (straight from global memory), their
//     R1-point transform, the twiddles w_n^(n2 k1), to shared memory;
//   R1 threads a line: R2 values, their R2-point transform, straight to global
//     memory (x: back to shared memory first, to part the two real lines of a
//     complex one).
//   x: real lines f[v][z][y][0..nx)   -> complex [v][z][y][0..nx/2]  (into the output)
//   y: complex lines along y, in place;  z: along z, in place, converted to FP64.
// A double-float complex value takes 16 bytes like a double2, so the output
// buffer holds the intermediate passes.  Axes other than 2^a 3^b <= 128 are
// not handled here (the caller falls back to cuFFT).
//
// Bound by the FP32 pipes: about 200 operations a value and axis (n = 96 as 8 x
// 12), 22 of them per complex addition.  The former passes (four in-place stages
// of radix 4, 4, 2, 3 through shared memory) spent as many again on addresses, and
// their conversions sent zeros and tiny values through the FP64 unit (60 % of
// its time in the x pass).  96 vectors of 96^3: 4.00 -> 1.79 ms a call (0.62 ms
// is the memory traffic of three passes at the copy rate); the Coulomb matrices
// of a 1 x 1 x 2 cell with three grids: 3.5 -> 1.95 ms of transforms.
#include <cmath>
#include <vector>

#include "dfloat.cuh"
#include "internal.cuh"

namespace isdf {
namespace {

constexpr int kMaxN = 128;

struct DC {
  DF re, im;
};
__device__ __forceinline__ DC dc_add(DC a, DC b) { return {df_add(a.re, b.re), df_add(a.im, b.im)}; }
__device__ __forceinline__ DC dc_sub(DC a, DC b) { return {df_sub(a.re, b.re), df_sub(a.im, b.im)}; }
// x y + sgn u v in double-float as one error-free sum of the two leading
// products, their exact rounding errors and the cross terms (the lo * lo
// terms, below 2^-48 of the result, are dropped as in df_mul)
__device__ __forceinline__ DF df_dot2(DF x, DF y, DF u, DF v, float sgn) {
  const float p = __fmul_rn(x.hi, y.hi), q = __fmul_rn(sgn * u.hi, v.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fadd_rn(e, __fmaf_rn(sgn * u.hi, v.hi, -q));
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  e = __fmaf_rn(sgn * u.hi, v.lo, e);
  e = __fmaf_rn(sgn * u.lo, v.hi, e);
  const DF s = two_sum(p, q);
  return quick_two_sum(s.hi, __fadd_rn(s.lo, e));
}
__device__ __forceinline__ DC dc_mul(DC a, DC b) {
  return {df_dot2(a.re, b.re, a.im, b.im, -1.0f), df_dot2(a.re, b.im, a.im, b.re, 1.0f)};
}
__device__ __forceinline__ DC dc_mul_mi(DC a) { return {a.im, df_neg(a.re)}; }  // a * (-i)
__device__ __forceinline__ DC dc_mul_pi(DC a) { return {df_neg(a.im), a.re}; }  // a * (+i)

__device__ __forceinline__ float4 dc_pack(DC a) { return make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }
__device__ __forceinline__ DC dc_unpack(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }

// x c for a constant c
__device__ __forceinline__ DC dc_scale(DC a, DF c) { return {df_mul(a.re, c), df_mul(a.im, c)}; }

// double-float constants from their FP64 values
__host__ __device__ constexpr DF dfc(double c) { return {float(c), float(c - double(float(c)))}; }
constexpr double kC8 = 0.70710678118654752440;                                   // cos(pi/4)
constexpr double kC16 = 0.92387953251128675613, kS16 = 0.38268343236508977173;   // pi/8
constexpr double kC9a = 0.76604444311897803520, kS9a = 0.64278760968653932632;   // 2 pi/9
constexpr double kC9b = 0.17364817766693034885, kS9b = 0.98480775301220805937;   // 4 pi/9
constexpr double kC9d = -0.93969262078590838405, kS9d = 0.34202014332566873304;  // 8 pi/9
// a exp(-i t) from cos t and sin t
__device__ __forceinline__ DC dc_rot(DC a, double c, double sn) { return dc_mul(a, {dfc(c), dfc(-sn)}); }
// a (1 - i) / sqrt(2) and a (-1 - i) / sqrt(2)
__device__ __forceinline__ DC dc_w8(DC a) { return dc_scale({df_add(a.re, a.im), df_sub(a.im, a.re)}, dfc(kC8)); }
__device__ __forceinline__ DC dc_w8_3(DC a) {
  return dc_scale({df_sub(a.im, a.re), df_neg(df_add(a.re, a.im))}, dfc(kC8));
}

// R-point transforms in registers, natural order in and out
__device__ __forceinline__ void dft(DC (&)[1]) {}
__device__ __forceinline__ void dft(DC (&a)[2]) {
  const DC t = dc_add(a[0], a[1]);
  a[1] = dc_sub(a[0], a[1]);
  a[0] = t;
}
__device__ __forceinline__ void dft(DC (&a)[3]) {  // w = exp(-2 pi i / 3) = -1/2 - i sqrt(3)/2
  const DF k = dfc(0.86602540378443864676);
  const DC b = dc_add(a[1], a[2]), c = dc_sub(a[1], a[2]);
  const DC t = {df_sub(a[0].re, df_half(b.re)), df_sub(a[0].im, df_half(b.im))};
  const DC kc = dc_scale(c, k);
  a[0] = dc_add(a[0], b);
  a[1] = dc_add(t, dc_mul_mi(kc));
  a[2] = dc_add(t, dc_mul_pi(kc));
}
__device__ __forceinline__ void dft(DC (&a)[4]) {
  const DC s02 = dc_add(a[0], a[2]), d02 = dc_sub(a[0], a[2]);
  const DC s13 = dc_add(a[1], a[3]), d13 = dc_sub(a[1], a[3]);
  a[0] = dc_add(s02, s13);
  a[2] = dc_sub(s02, s13);
  a[1] = dc_add(d02, dc_mul_mi(d13));
  a[3] = dc_add(d02, dc_mul_pi(d13));
}
// R1 x R2 coprime: n = R2 n1 + R1 n2, k = (k mod R1, k mod R2), no twiddles
template <int R1, int R2>
__device__ __forceinline__ void dft_coprime(DC (&a)[R1 * R2]) {
  constexpr int N = R1 * R2;
  DC t[R2][R1];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) t[n2][n1] = a[(R2 * n1 + R1 * n2) % N];
    dft(t[n2]);
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    DC u[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) u[n2] = t[n2][k1];
    dft(u);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2)
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (k % R1 == k1 && k % R2 == k2) a[k] = u[k2];
  }
}
__device__ __forceinline__ void dft(DC (&a)[6]) { dft_coprime<2, 3>(a); }
__device__ __forceinline__ void dft(DC (&a)[12]) { dft_coprime<4, 3>(a); }
__device__ __forceinline__ void dft(DC (&a)[8]) {
  DC e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
  dft(e);
  dft(o);
  o[1] = dc_w8(o[1]);
  o[2] = dc_mul_mi(o[2]);
  o[3] = dc_w8_3(o[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k] = dc_add(e[k], o[k]), a[k + 4] = dc_sub(e[k], o[k]);
}
// N = R R: n = R n1 + n2, k = k1 + R k2, twiddles w_N^(n2 k1)
__device__ __forceinline__ DC dc_w9(DC a, int e) {
  return e == 1 ? dc_rot(a, kC9a, kS9a) : e == 2 ? dc_rot(a, kC9b, kS9b) : e == 4 ? dc_rot(a, kC9d, kS9d) : a;
}
__device__ __forceinline__ DC dc_w16(DC a, int e) {
  return e == 1   ? dc_rot(a, kC16, kS16)
         : e == 2 ? dc_w8(a)
         : e == 3 ? dc_rot(a, kS16, kC16)
         : e == 4 ? dc_mul_mi(a)
         : e == 6 ? dc_w8_3(a)
         : e == 9 ? dc_rot(a, -kC16, -kS16)
                  : a;
}
template <int R, class W>
__device__ __forceinline__ void dft_square(DC (&a)[R * R], W tw) {
  DC t[R][R];
#pragma unroll
  for (int n2 = 0; n2 < R; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < R; ++n1) t[n2][n1] = a[R * n1 + n2];
    dft(t[n2]);
  }
#pragma unroll
  for (int k1 = 0; k1 < R; ++k1) {
    DC u[R];
#pragma unroll
    for (int n2 = 0; n2 < R; ++n2) u[n2] = tw(t[n2][k1], n2 * k1);
    dft(u);
#pragma unroll
    for (int k2 = 0; k2 < R; ++k2) a[k1 + R * k2] = u[k2];
  }
}
__device__ __forceinline__ void dft(DC (&a)[9]) {
  dft_square<3>(a, [](DC x, int e) { return dc_w9(x, e); });
}
__device__ __forceinline__ void dft(DC (&a)[16]) {
  dft_square<4>(a, [](DC x, int e) { return dc_w16(x, e); });
}

struct FftPass {
  int n, r1, r2;
  int lpb;                  // complex lines per block
  int64_t nlines;           // complex lines (x: two real lines of one vector make one)
  int64_t nreal, npair;     // x: real and complex lines per vector
  // line l starts at (l / lin) * lso + (l % lin) * lsi (lin 0: l * lsi); element e at + e * es
  // (all in values of the input / output arrays)
  int64_t lin, lso, lsi, es;
  int nout;                 // elements written per line (x pass: n / 2 + 1)
  const float4* tw;         // exp(-2 pi i k / n), k < n
  const double* in_real;    // x pass input (real), else nullptr
  float4* io;               // complex data (double-float), in/out
  double2* out64;           // last pass: FP64 output (same buffer), else nullptr
};

// floor(x / d) for x < 2^16, 1 <= d <= 128: with M = ceil(2^32 / d) the high
// word of x M is exact (the rounding error x (M - 2^32/d) / 2^32 < 2^-16 stays
// below the gap 1/d between x/d and the next integer).  M = 0 encodes d = 1.
struct FastDiv {
  unsigned int d, M;
};
__host__ __device__ inline FastDiv fast_div(unsigned int d) {
  return {d, d == 1 ? 0u : (unsigned int)((0xFFFFFFFFull + d) / d)};
}
__device__ __forceinline__ int fdiv(int x, FastDiv f) { return f.M ? int(__umulhi(unsigned(x), f.M)) : x; }

__device__ __forceinline__ int64_t line_base(const FftPass& P, int64_t l) {
  return P.lin ? (l / P.lin) * P.lso + (l % P.lin) * P.lsi : l * P.lsi;
}

// Real lines of complex line c (x pass): a vector's own, so that no rounding of
// one vector reaches another; an odd last line is alone.
struct RealPair {
  int64_t line;
  bool two;
};
__device__ __forceinline__ RealPair real_pair(const FftPass& P, int64_t c) {
  const int64_t v = c / P.npair, p = c - v * P.npair;
  return {v * P.nreal + 2 * p, 2 * p + 1 < P.nreal};
}

// shared memory of a line: value n2 of transform k1 at k1 * row + n2, lines ld apart (both odd: the
// 16-byte accesses of eight neighbouring threads fall in different banks either way)
__host__ __device__ constexpr int fft_row(int r2) { return r2 | 1; }
__host__ __device__ constexpr int fft_ld(int r1, int r2) { return (r1 * fft_row(r2)) | 1; }

// First half: thread tasks (line, n2)
template <int R1>
__device__ __forceinline__ void fft_first(const FftPass& P, float4* buf, const float4* tws, int64_t l0, int lines) {
  const int R2 = P.r2, ld = fft_ld(R1, R2), row = fft_row(R2);
  const bool real = P.in_real != nullptr;
  const FastDiv dr = fast_div(R2), dl = fast_div(lines);
  for (int idx = threadIdx.x; idx < lines * R2; idx += blockDim.x) {
    // neighbouring threads: neighbouring elements of a contiguous line, else neighbouring lines
    int li, n2;
    if (real) li = fdiv(idx, dr), n2 = idx - li * R2;
    else n2 = fdiv(idx, dl), li = idx - n2 * lines;
    DC a[R1];
    if (real) {
      const RealPair q = real_pair(P, l0 + li);
      const double* fa = P.in_real + q.line * P.lsi + n2;
      const bool two = q.two;
      // all loads before the first conversion, whose branches would part them
      double vr[R1], vi[R1];
#pragma unroll
      for (int t = 0; t < R1; ++t) vr[t] = fa[t * R2], vi[t] = two ? fa[P.lsi + t * R2] : 0.0;
#pragma unroll
      for (int t = 0; t < R1; ++t) a[t].re = df_from_double(vr[t]), a[t].im = df_from_double(vi[t]);
    } else {
      const float4* x = P.io + line_base(P, l0 + li) + n2 * P.es;
      const int64_t step = R2 * P.es;
#pragma unroll
      for (int t = 0; t < R1; ++t) a[t] = dc_unpack(x[t * step]);
    }
    dft(a);
    float4* y = buf + li * ld + n2;
    y[0] = dc_pack(a[0]);
#pragma unroll
    for (int k = 1; k < R1; ++k) y[k * row] = dc_pack(n2 ? dc_mul(a[k], dc_unpack(tws[n2 * k])) : a[k]);
  }
}

// Second half: thread tasks (line, k1); transform k = k1 + r1 k2
template <int R2>
__device__ __forceinline__ void fft_second(const FftPass& P, float4* buf, int64_t l0, int lines) {
  const int R1 = P.r1, ld = fft_ld(R1, R2), row = fft_row(R2);
  const bool real = P.in_real != nullptr;
  const FastDiv dr = fast_div(R1), dl = fast_div(lines);
  for (int idx = threadIdx.x; idx < lines * R1; idx += blockDim.x) {
    int li, k1;
    if (real) li = fdiv(idx, dr), k1 = idx - li * R1;
    else k1 = fdiv(idx, dl), li = idx - k1 * lines;
    float4* y = buf + li * ld + k1 * row;
    DC a[R2];
#pragma unroll
    for (int t = 0; t < R2; ++t) a[t] = dc_unpack(y[t]);
    dft(a);
    if (real) {
#pragma unroll
      for (int t = 0; t < R2; ++t) y[t] = dc_pack(a[t]);
    } else {
      const int64_t base = line_base(P, l0 + li) + k1 * P.es, step = R1 * P.es;
      if (P.out64) {
#pragma unroll
        for (int t = 0; t < R2; ++t)
          P.out64[base + t * step] = make_double2(df_to_double(a[t].re), df_to_double(a[t].im));
      } else {
#pragma unroll
        for (int t = 0; t < R2; ++t) P.io[base + t * step] = dc_pack(a[t]);
      }
    }
  }
}

// BIG: axes with a 16-point half (n = 128), whose registers would halve the
// occupancy of the others
constexpr int kFftThreads = 128;
template <bool BIG>
__global__ void __launch_bounds__(kFftThreads, BIG ? 2 : 4) k_fft_pass(FftPass P) {
  extern __shared__ float4 sm[];
  __shared__ float4 tws[kMaxN];
  const bool real = P.in_real != nullptr;
  const int64_t l0 = int64_t(blockIdx.x) * P.lpb;
  const int lines = int(P.nlines - l0 < P.lpb ? P.nlines - l0 : P.lpb);
  for (int i = threadIdx.x; i < P.n; i += blockDim.x) tws[i] = P.tw[i];
  __syncthreads();
  if constexpr (BIG) {
    fft_first<16>(P, sm, tws, l0, lines);
  } else {
    switch (P.r1) {
      case 1: fft_first<1>(P, sm, tws, l0, lines); break;
      case 2: fft_first<2>(P, sm, tws, l0, lines); break;
      case 3: fft_first<3>(P, sm, tws, l0, lines); break;
      case 4: fft_first<4>(P, sm, tws, l0, lines); break;
      case 6: fft_first<6>(P, sm, tws, l0, lines); break;
      case 8: fft_first<8>(P, sm, tws, l0, lines); break;
      default: fft_first<9>(P, sm, tws, l0, lines); break;
    }
  }
  __syncthreads();
  if constexpr (BIG) {
    fft_second<8>(P, sm, l0, lines);
  } else {
    switch (P.r2) {
      case 1: fft_second<1>(P, sm, l0, lines); break;
      case 2: fft_second<2>(P, sm, l0, lines); break;
      case 3: fft_second<3>(P, sm, l0, lines); break;
      case 4: fft_second<4>(P, sm, l0, lines); break;
      case 6: fft_second<6>(P, sm, l0, lines); break;
      case 8: fft_second<8>(P, sm, l0, lines); break;
      case 9: fft_second<9>(P, sm, l0, lines); break;
      default: fft_second<12>(P, sm, l0, lines); break;
    }
  }
  if (!real) return;
  __syncthreads();
  // Z = F_a + i F_b with F_a, F_b Hermitian:  F_a = (Z_k + conj Z_{n-k}) / 2,
  // F_b = -i (Z_k - conj Z_{n-k}) / 2
  const int nout = P.nout, ld = fft_ld(P.r1, P.r2), row = fft_row(P.r2);
  const FastDiv dout = fast_div(nout), d1 = fast_div(P.r1);
  auto at = [&](int li, int k) {  // transform k = k1 + r1 k2
    const int k2 = fdiv(k, d1);
    return dc_unpack(sm[li * ld + (k - k2 * P.r1) * row + k2]);
  };
  for (int idx = threadIdx.x; idx < lines * nout; idx += blockDim.x) {
    const int li = fdiv(idx, dout), e = idx - li * nout;
    const DC zk = at(li, e), zc = at(li, e == 0 ? 0 : P.n - e);
    const DC w = {zc.re, df_neg(zc.im)};
    const DC sum = dc_add(zk, w), d = dc_sub(zk, w);
    const RealPair q = real_pair(P, l0 + li);
    float4* out = P.io + q.line * nout + e;
    out[0] = dc_pack({df_half(sum.re), df_half(sum.im)});
    if (q.two) out[nout] = dc_pack({df_half(d.im), df_half(df_neg(d.re))});
  }
}

// n = r1 r2 with halves of at most 9 and 12 points (16 and 8 for 128)
constexpr int kAxes[][3] = {{1, 1, 1},  {2, 1, 2},  {3, 1, 3},  {4, 2, 2},  {6, 2, 3},  {8, 2, 4},  {9, 3, 3},   {12, 3, 4},
                            {16, 4, 4}, {18, 3, 6}, {24, 4, 6}, {27, 3, 9}, {32, 4, 8}, {36, 6, 6}, {48, 6, 8},  {54, 6, 9},
                            {64, 8, 8}, {72, 8, 9}, {81, 9, 9}, {96, 8, 12}, {108, 9, 12}, {128, 16, 8}};
bool split_axis(int n, int* r1, int* r2) {
  for (const auto& t : kAxes)
    if (t[0] == n) return *r1 = t[1], *r2 = t[2], true;
  return false;
}

// Lines per block: whole rounds of the 128 threads in both halves for the usual
// sizes, and at most about 64 KB
constexpr int fft_lines(int n) { return n >= 48 ? 32 : n >= 24 ? 64 : 128; }
constexpr int fft_smem(int n, int r1, int r2) { return fft_lines(n) * fft_ld(r1, r2) * int(sizeof(float4)); }
// the most that any axis of a kernel's needs
constexpr int fft_max_smem(bool big) {
  int m = 0;
  for (const auto& t : kAxes)
    if ((t[1] == 16) == big && fft_smem(t[0], t[1], t[2]) > m) m = fft_smem(t[0], t[1], t[2]);
  return m;
}

}  // namespace

bool rfft3_df_supported(int nx, int ny, int nz) {
  int a, b;
  return split_axis(nx, &a, &b) && split_axis(ny, &a, &b) && split_axis(nz, &a, &b);
}

// f: batch x (nz ny nx) FP64, S: batch x (nz ny (nx/2+1)) double2 (device);
// tw: device scratch of 2 (nx + ny + nz) float4 (twiddle tables).
isdf_status rfft3_df(Plan* p, const double* f, int nx, int ny, int nz, int64_t batch, double2* S, cudaStream_t s) {
  if (!rfft3_df_supported(nx, ny, nz)) return fail(p, ISDF_ERR_ARG, "double-float transform: unsupported grid");
  if (batch <= 0) return ISDF_OK;
  const int nxh = nx / 2 + 1;
  // twiddle tables exp(-2 pi i k / n) as double-float, from FP64
  std::vector<float> tw(size_t(4) * (nx + ny + nz));
  size_t o = 0;
  int64_t toff[3];
  const int ns[3] = {nx, ny, nz};
  for (int a = 0; a < 3; ++a) {
    toff[a] = int64_t(o / 4);
    for (int k = 0; k < ns[a]; ++k) {
      const double th = -2.0 * 3.14159265358979323846 * double(k) / double(ns[a]);
      const double c = std::cos(th), sn = std::sin(th);
      const float ch = float(c), sh = float(sn);
      tw[o++] = ch;
      tw[o++] = float(c - double(ch));
      tw[o++] = sh;
      tw[o++] = float(sn - double(sh));
    }
  }
  float4* dtw = nullptr;
  isdf_status st;
  const auto release = [&] { p ? dfree(dtw) : scratch_free(dtw, s); };
  if (p) {
    if ((st = dalloc_t(p, &dtw, tw.size() / 4, "transform twiddles"))) return st;
  } else {
    const cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&dtw), sizeof(float) * tw.size(), s);
    if (e != cudaSuccess)
      return fail(p, e == cudaErrorMemoryAllocation ? ISDF_ERR_OOM : ISDF_ERR_CUDA,
                  std::string("transform twiddles: ") + cudaGetErrorString(e));
  }
  if ((st = cuda_check(p, cudaMemcpyAsync(dtw, tw.data(), sizeof(float) * tw.size(), cudaMemcpyHostToDevice, s),
                       "twiddle copy"))) {
    release();
    return st;
  }
  float4* io = reinterpret_cast<float4*>(S);
  const int64_t nq = int64_t(nz) * ny * nxh;
  cudaError_t failed = cudaSuccess;  // the first launch that was refused: its pass is missing
  auto launch = [&](FftPass P) {
    if (failed != cudaSuccess) return;
    split_axis(P.n, &P.r1, &P.r2);
    P.lpb = fft_lines(P.n);
    const int64_t blocks = (P.nlines + P.lpb - 1) / P.lpb;
    const bool big = P.r1 == 16;
    auto kernel = big ? k_fft_pass<true> : k_fft_pass<false>;
    // the limit belongs to the kernel, not to this call: every caller sets the
    // same value, so that no thread lowers it under another's launch
    failed = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  big ? fft_max_smem(true) : fft_max_smem(false));
    if (failed != cudaSuccess) return;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(kFftThreads);
    cfg.dynamicSmemBytes = size_t(fft_smem(P.n, P.r1, P.r2));
    cfg.stream = s;
    failed = cudaLaunchKernelEx(&cfg, kernel, P);
    count_launches(1);
  };
  // x: lines (v, z, y), contiguous
  FftPass P{};
  P.n = nx;
  P.nreal = int64_t(nz) * ny;
  P.npair = (P.nreal + 1) / 2;
  P.nlines = batch * P.npair;
  P.lin = 0;
  P.lsi = nx;
  P.es = 1;
  P.nout = nxh;
  P.tw = dtw + toff[0];
  P.in_real = f;
  P.io = io;
  launch(P);
  // y: lines (v, z, qx), element stride nxh, in place
  FftPass Q{};
  Q.n = ny;
  Q.nlines = batch * nz * nxh;
  Q.lin = nxh;
  Q.lso = int64_t(ny) * nxh;
  Q.lsi = 1;
  Q.es = nxh;
  Q.nout = ny;
  Q.tw = dtw + toff[1];
  Q.io = io;
  launch(Q);
  // z: lines (v, qy, qx), element stride ny nxh, in place, FP64 out
  FftPass R{};
  R.n = nz;
  R.nlines = batch * ny * nxh;
  R.lin = int64_t(ny) * nxh;
  R.lso = nq;
  R.lsi = 1;
  R.es = int64_t(ny) * nxh;
  R.nout = nz;
  R.tw = dtw + toff[2];
  R.io = io;
  R.out64 = S;
  launch(R);
  release();
  if (failed != cudaSuccess) cudaGetLastError();  // reported here
  return cuda_check(p, failed, "double-float transform");
}

}  // namespace isdf
