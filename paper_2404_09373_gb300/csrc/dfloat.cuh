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
// FP64 and rounded once to FP32.  Below 2^-73 lo runs into FP32's subnormals
// (reached through a second power of two), below 2^-126 hi does and nothing is
// left for lo; only values above 2^125 take the FP64 route.
__device__ __forceinline__ DF df_from_double(double x) {
  const uint64_t b = uint64_t(__double_as_longlong(x));
  const int E = int((b >> 52) & 0x7FF);
  if (E > 1148) {
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - double(hi))};
  }
  const uint32_t sign = uint32_t(b >> 32) & 0x80000000u;
  if (E < 897) {  // |x| < 2^-126
    uint32_t q = 0u;  // |x| in units of 2^-149, to the nearest (ties to even)
    if (E > 872) {
      const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
      const int r = 926 - E;
      q = uint32_t((m + ((1ull << (r - 1)) - 1ull) + ((m >> r) & 1ull)) >> r);
    }
    return {__uint_as_float(q | sign), 0.0f};
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

// r = 1 / sqrt(d) and s = sqrt(d) for finite d > 0.  r: FP32 estimate of the
// significand's root and one step of the third-order iteration r (1 + e/2 + 3 e^2 /
// 8), e = 1 - d r^2 (the Taylor series of (1 - e)^-1/2): from 2^-22 to rounding error
// in four dependent FP64 operations instead of the forty of a square root and a
// division.  s: d r and one correction by its residual.  Both on the significand,
// scaled back by its exponent, so that no residual of a tiny d runs into the
// subnormal numbers.
struct Root64 {
  double r, s;
};
__device__ __forceinline__ Root64 root64(double d) {
  const long long b = __double_as_longlong(d);
  const int E = int((b >> 52) & 0x7FF);
  if (E == 0) {  // subnormal
    const double s = sqrt(d);
    return {1.0 / s, s};
  }
  const int h = (E - 1023) >> 1;  // d = m 4^h, m in [1, 4)
  const double m = __longlong_as_double(b - ((long long)(2 * h) << 52));
  const int odd = (E - 1023) & 1;
  const float mf = __int_as_float(((127 + odd) << 23) | int((b >> 29) & 0x7FFFFF));
  const double r0 = f32_to_f64(rsqrtf(mf));
  const double t = m * r0;
  const double e = fma(-t, r0, 1.0);
  const double r = fma(r0 * e, fma(0.375, e, 0.5), r0);
  const double s0 = m * r, s = fma(fma(-s0, s0, m), 0.5 * r, s0);
  const long long hs = (long long)h << 52;
  return {__longlong_as_double(__double_as_longlong(r) - hs), __longlong_as_double(__double_as_longlong(s) + hs)};
}

// 1 / sqrt(d) as a double-float, FP32 operations only: the same iteration.  Its
// residual e = 1 - m r^2 is kept to 2^-70 or so: m's 53 bits in three parts, every
// product of two parts above 2^-50 with its rounding error, so that the result
// carries little more than a double-float's own rounding: 2^-49.0 at most over
// [1, 4) (1 / sqrt(d) in FP64 rounded to a pair: 2^-48.9; with the residual in one
// pair: 2^-47.1).
__device__ __forceinline__ DF df_rsqrt(double d) {
  const long long b = __double_as_longlong(d);
  const int E = int((b >> 52) & 0x7FF);
  const int h = (E - 1023) >> 1;  // d = m 4^h, m in [1, 4)
  if (E == 0 || h < -120 || h > 120) return df_from_double(1.0 / sqrt(d));
  const DF m = df_from_double(__longlong_as_double(b - ((long long)(2 * h) << 52)));
  // what m.lo leaves of the low 29 bits (below 2^-48)
  const int m29 = int(uint32_t(b) & 0x1FFFFFFFu), i29 = m29 - ((m29 >> 28) << 29);
  const float rest = __int2float_rn(i29 - __float2int_rn(__int2float_rn(i29))) * ((E - 1023) & 1 ? 0x1p-51f : 0x1p-52f);
  const float r = rsqrtf(m.hi);
  // m r = p + (u.hi + u.lo + te)
  const float p = __fmul_rn(m.hi, r), pe = __fmaf_rn(m.hi, r, -p);
  const float t = __fmul_rn(m.lo, r), te = __fmaf_rn(rest, r, __fmaf_rn(m.lo, r, -t));
  const DF u = two_sum(pe, t);
  // m r^2 = q + qe + v + ve
  const float q = __fmul_rn(p, r), qe = __fmaf_rn(p, r, -q);
  const float v = __fmul_rn(u.hi, r), ve = __fmaf_rn(__fadd_rn(u.lo, te), r, __fmaf_rn(u.hi, r, -v));
  const DF e1 = two_sum(__fsub_rn(1.0f, q), -qe);  // 1 - q is exact
  DF e = two_sum(e1.hi, -v);
  e.lo = __fadd_rn(e.lo, __fsub_rn(e1.lo, ve));
  const float hr = 0.5f * r, c = __fmul_rn(hr, e.hi);
  const float cl = __fmaf_rn(hr, e.hi, -c) + __fmaf_rn(hr, e.lo, hr * (0.75f * e.hi * e.hi));
  const DF s = two_sum(r, c);
  const DF x = quick_two_sum(s.hi, __fadd_rn(s.lo, cl));
  const float sc = __int_as_float((127 - h) << 23);
  return {x.hi * sc, x.lo * sc};
}

}  // namespace
}  // namespace isdf
