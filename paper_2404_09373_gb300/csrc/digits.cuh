// BF16 digit planes of FP64 values (the operands of the tensor-core products):
// rounding to the row's scale, digit extraction, and the place of a digit in the
// tiled operand.  Integer and FP32 operations only, off the narrow FP64 unit.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

#include "internal.cuh"

namespace isdf {
namespace {

// round(x * 2^shift) to the nearest integer (ties to even) with integer
// operations only; |result| < 2^62 is guaranteed by the caller's scaling.
// Right shifts round by adding (half - 1 + the kept low bit) before the shift.
__device__ __forceinline__ long long round_scaled(double x, int shift) {
  const uint64_t b = uint64_t(__double_as_longlong(x));
  const int E = int((b >> 52) & 0x7FF);
  const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (uint64_t(E != 0) << 52);
  const int r = 1075 - (E ? E : 1) - shift;  // value = m * 2^-r
  uint64_t q;
  if (r > 0) {
    q = r < 64 ? (m + ((1ull << (r - 1)) - 1ull) + ((m >> r) & 1ull)) >> r : 0ull;
  } else {
    q = m << -r;
  }
  return (b >> 63) ? -(long long)q : (long long)q;
}

// BF16 bits of a small integer d (|d| <= 2^8): 1.5 * 2^23 + d is exact in
// FP32 (unit spacing), subtracting 1.5 * 2^23 leaves d exactly, and d has at
// most 8 significant bits, so the upper half of its FP32 pattern is its BF16
// pattern.  Integer and FP32 operations only.
__device__ __forceinline__ uint32_t bf16_bits_of_small(int d) {
  return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f);
}

// Digits of 8 consecutive k values of one row, 16 bytes per slice at
// out + s * tile_elems.  With X = round(x 2^shift) the balanced digits
// (in [-64, 63], the top one takes the rest, |d_0| <= 128) are the base-128
// digits of X + sum_p 64 128^p less 64, so every digit is a 7-bit field of one
// integer and no digit waits for the one below it; two fields go through
// BF16 at once, 0x4300 | f being the pattern of 128 + f and the difference to
// 192 exact.
template <int S>
__device__ __forceinline__ void oz_digits8(const double (&v)[8], int shift, int64_t tile_elems,
                                           __nv_bfloat16* __restrict__ out) {
  constexpr long long bias = 64ll * (((1ll << (7 * (S - 1))) - 1ll) / 127ll);
  uint32_t w0[8];  // fields 0..3 (the least significant digits)
  int w1[8];       // fields 4.. and the top digit (signed)
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const long long X = round_scaled(v[u], shift) + bias;
    w0[u] = uint32_t(X) & 0x0FFFFFFFu;
    w1[u] = int(X >> 28);
  }
  const __nv_bfloat162 c192 = __floats2bfloat162_rn(192.0f, 192.0f);
#pragma unroll
  for (int s = S - 1; s >= 0; --s) {
    uint32_t r[4];
    const int p = S - 1 - s;  // field position, 7 p bits up
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      if (s == 0) {
        const int sh = 7 * (S - 1) - 28;
        r[h] = __byte_perm(bf16_bits_of_small(w1[2 * h] >> sh), bf16_bits_of_small(w1[2 * h + 1] >> sh), 0x7632);
      } else {
        const int sh = 7 * (p & 3);
        const uint32_t a = p < 4 ? w0[2 * h] : uint32_t(w1[2 * h]);
        const uint32_t b = p < 4 ? w0[2 * h + 1] : uint32_t(w1[2 * h + 1]);
        const uint32_t bu = sh <= 16 ? b << (16 - sh) : b >> (sh - 16);
        const uint32_t t = ((a >> sh) & 0x7Fu) | (bu & 0x7F0000u) | 0x43004300u;
        const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&t), c192);
        r[h] = *reinterpret_cast<const uint32_t*>(&d);
      }
    }
    *reinterpret_cast<uint4*>(out + int64_t(s) * tile_elems) = make_uint4(r[0], r[1], r[2], r[3]);
  }
}

// Element offset of the 8 values (row rr of a tile, 8-wide k group kc of it) in one slice of a tile.
__device__ __forceinline__ int oz_inner(int rr, int kc) { return (rr >> 3) * (8 * kOzBK) + kc * 64 + (rr & 7) * 8; }

// Digits (8 slices) of columns [c0, c1) of row t of a 128-row-tile operand, whole
// groups of 8 columns from the first one touched: column c at x[c * ldx], zero
// from c1 on.  e: the row's scale; kst: k tiles per row tile.
__device__ __forceinline__ void oz_append_row(const double* __restrict__ x, int64_t ldx, int c0, int c1, int e, int64_t t,
                                              int64_t kst, void* tiles) {
  constexpr int S = 8;
  const int64_t tile_elems = 128 * kOzBK;
  for (int g = c0 / 8; g * 8 < c1; ++g) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = g * 8 + u < c1 ? x[int64_t(g * 8 + u) * ldx] : 0.0;
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(tiles) +
                         (((t >> 7) * kst + g / (kOzBK / 8)) * S) * tile_elems + oz_inner(int(t & 127), g % (kOzBK / 8));
    oz_digits8<S>(v, 7 * S - e, tile_elems, out);
  }
}

}  // namespace
}  // namespace isdf
