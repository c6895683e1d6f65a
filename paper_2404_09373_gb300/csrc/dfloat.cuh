// Double-float arithmetic: a value is a pair of FP32 numbers (hi, lo) with
// hi + lo the represented number (about 48 significant bits).  Sums use an
// error-free two-sum and products an FMA-based two-product, so the work runs
// on the FP32 pipes, tens of times the FP64 rate on this GPU; conversions
// from and to FP64 use integer operations and at most one FP64 addition.
#pragma once

#include <cstdint>

namespace isdf {
namespace {

struct DF {
  float hi, lo;
};

// Error-free transformations with explicitly rounded operations (the
// compiler must not contract them into FMAs or reassociate them).
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ DF quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF df_add(DF x, DF y) {
  DF s = two_sum(x.hi, y.hi);
  s.lo = __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo));
  return quick_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ DF df_neg(DF x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ DF df_sub(DF x, DF y) { return df_add(x, df_neg(y)); }
__device__ __forceinline__ DF df_mul(DF x, DF y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);  // exact error of the product
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return quick_two_sum(p, e);
}
__device__ __forceinline__ DF df_half(DF x) { return {__fmul_rn(0.5f, x.hi), __fmul_rn(0.5f, x.lo)}; }


// Conversions between FP64 and double-float with integer and FP32 operations, so
// that they stay off the narrow FP64 unit.  hi is x's significand rounded to 24
// bits (the round bit added into the exponent|significand field carries
// correctly); lo = x - hi is the signed remainder of the low 29 bits, exact in
// FP64 and rounded once to FP32.  Below 2^-73 lo, and below 2^-126 hi, run
// into FP32's subnormals (both reached through a second power of two); only
// values above 2^125 take the FP64 route.
__device__ __forceinline__ DF df_from_double(double x) {
  const uint64_t b = uint64_t(__double_as_longlong(x));
  const int E = int((b >> 52) & 0x7FF);
  if (E > 1148) {
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - double(hi))};
  }
  const uint32_t sign = uint32_t(b >> 32) & 0x80000000u;
  if (E < 897) {  // |x| < 2^-126
    const float m = __uint_as_float(0x3F800000u | (uint32_t(b >> 29) & 0x7FFFFFu));
    const float hi = E > 860 ? __fmul_rn(__fmul_rn(m, 0x1p-100f), __uint_as_float(uint32_t(E - 796) << 23)) : 0.0f;
    return {__uint_as_float(__float_as_uint(hi) | sign), 0.0f};
  }
  const uint32_t m29 = uint32_t(b) & 0x1FFFFFFFu;
  const uint32_t up = m29 >> 28;
  const uint32_t hb = ((uint32_t(E - 896) << 23) | (uint32_t(b >> 29) & 0x7FFFFFu)) + up;
  const int q = E >= 950 ? 0 : 100;  // 2^(E - 1075), in two factors below 2^-125
  float lo = __int2float_rn(int(m29) - int(up << 29)) * __uint_as_float(uint32_t(E - 948 + q) << 23);
  if (q) lo = __fmul_rn(lo, 0x1p-100f);
  return {__uint_as_float(hb | sign), sign ? -lo : lo};
}

// FP32 value as FP64 bits, exact
__device__ __forceinline__ double f32_to_f64(float f) {
  const uint32_t b = __float_as_uint(f), m = b & 0x7FFFFFu;
  const uint32_t ef = (b >> 23) & 0xFFu;
  const uint64_t sign = uint64_t(b & 0x80000000u) << 32;
  uint64_t bits = (uint64_t(ef + 896u) << 52) | (uint64_t(m) << 29);
  if (ef == 0u) {  // zero, or a subnormal: m 2^-149
    const int lz = __clz(int(m));
    bits = m ? (uint64_t(905u - uint32_t(lz)) << 52) + ((uint64_t(m) << (lz + 21)) & 0xFFFFFFFFFFFFFull) : 0ull;
  } else if (ef == 0xFFu) {
    bits = (0x7FFull << 52) | (uint64_t(m) << 29);
  }
  return __longlong_as_double((long long)(sign | bits));
}
__device__ __forceinline__ double df_to_double(DF x) { return f32_to_f64(x.hi) + f32_to_f64(x.lo); }

// 1 / sqrt(d) for finite d > 0: FP32 estimate of the significand's root and one
// step of the third-order iteration r (1 + e/2 + 3 e^2 / 8), e = 1 - d r^2 (the
// Taylor series of (1 - e)^-1/2): from 2^-22 to rounding error in four dependent
// FP64 operations instead of the forty of a square root and a division.
__device__ __forceinline__ double rsqrt64(double d) {
  const long long b = __double_as_longlong(d);
  int E = int((b >> 52) & 0x7FF);
  if (E == 0) return 1.0 / sqrt(d);  // subnormal
  const int h = (E - 1023) >> 1;     // d = m 4^h, m in [1, 4)
  const double m = __longlong_as_double(b - ((long long)(2 * h) << 52));
  const int odd = (E - 1023) & 1;
  const float mf = __int_as_float(((127 + odd) << 23) | int((b >> 29) & 0x7FFFFF));
  const double r0 = f32_to_f64(rsqrtf(mf));
  const double t = m * r0;
  const double e = fma(-t, r0, 1.0);
  const double r = fma(r0 * e, fma(0.375, e, 0.5), r0);
  return __longlong_as_double(__double_as_longlong(r) - ((long long)h << 52));
}

// 1 / sqrt(d) as a double-float, FP32 operations only: the same iteration with
// the residual e = 1 - m r0^2 and its correction carried as pairs.
__device__ __forceinline__ DF df_rsqrt(double d) {
  const long long b = __double_as_longlong(d);
  const int E = int((b >> 52) & 0x7FF);
  const int h = (E - 1023) >> 1;  // d = m 4^h, m in [1, 4)
  if (E == 0 || h < -120 || h > 120) return df_from_double(1.0 / sqrt(d));
  const DF m = df_from_double(__longlong_as_double(b - ((long long)(2 * h) << 52)));
  const float r = rsqrtf(m.hi);
  const float p = __fmul_rn(m.hi, r);
  const float pe = __fmaf_rn(m.lo, r, __fmaf_rn(m.hi, r, -p));
  const float q = __fmul_rn(p, r);
  const float qe = __fmaf_rn(pe, r, __fmaf_rn(p, r, -q));
  const DF e = two_sum(__fsub_rn(1.0f, q), -qe);  // 1 - q is exact
  const float hr = 0.5f * r, c = __fmul_rn(hr, e.hi);
  const float cl = __fmaf_rn(hr, e.hi, -c) + __fmaf_rn(hr, e.lo, hr * (0.75f * e.hi * e.hi));
  const DF s = two_sum(r, c);
  const DF x = quick_two_sum(s.hi, __fadd_rn(s.lo, cl));
  const float sc = __int_as_float((127 - h) << 23);
  return {x.hi * sc, x.lo * sc};
}

// sqrt(d) from r = rsqrt64(d)
__device__ __forceinline__ double sqrt_from(double d, double r) {
  const double s = d * r;
  return fma(fma(-s, s, d), 0.5 * r, s);
}

}  // namespace
}  // namespace isdf
