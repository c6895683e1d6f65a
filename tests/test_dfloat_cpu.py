"""Double-float helpers (csrc/dfloat.cuh) compiled for the host: the operations are IEEE single and double precision
either way; rsqrtf, accurate to 2 units in the last place on the GPU, is given every error from -2 to 2 units.

Bounds.  A pair's own rounding is 2^-49 relative (hi 24 bits, lo 24 bits of the rest).
df_rsqrt: that and 2^-52, what FP64's square root and division leave.
root64: r 2^-53 for the last rounding and half of that for the rounding in its residual, s one rounding, 2^-53; terms
below 2^-62 in both."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09373_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
template <class T, class F> static T bits_as(F f) { T t; std::memcpy(&t, &f, sizeof t); return t; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static long long __double_as_longlong(double x) { return bits_as<long long>(x); }
static double __longlong_as_double(long long x) { return bits_as<double>(x); }
static unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
static float __uint_as_float(unsigned x) { return bits_as<float>(x); }
static float __int_as_float(int x) { return bits_as<float>(x); }
static float __double2float_rn(double x) { return float(x); }
static float __int2float_rn(int x) { return float(x); }
static int __float2int_rn(float x) { return int(std::nearbyint(x)); }
static int __clz(int x) { return x ? __builtin_clz(unsigned(x)) : 32; }
static int off = 0;
static float rsqrtf(float x) { return __int_as_float(bits_as<int>(float(1.0 / std::sqrt(double(x)))) + off); }
using std::sqrt;
#include "dfloat.cuh"
using namespace isdf;
extern "C" {
void t_rsqrt(const double* d, int n, int ulps, float* hi, float* lo, double* r, double* s) {
  off = ulps;
  for (int i = 0; i < n; ++i) {
    const DF x = df_rsqrt(d[i]);
    hi[i] = x.hi, lo[i] = x.lo;
    const Root64 q = root64(d[i]);
    r[i] = q.r, s[i] = q.s;
  }
}
void t_pair(const double* x, int n, float* hi, float* lo, double* back) {
  for (int i = 0; i < n; ++i) {
    const DF p = df_from_double(x[i]);
    hi[i] = p.hi, lo[i] = p.lo;
    back[i] = df_to_double(p);
  }
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("dfloat")
    (d / "df.cpp").write_text(SOURCE)
    so = str(d / "libdf.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC, str(d / "df.cpp"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
@pytest.mark.parametrize("lo,hi", [(0, 2), (-60, 60), (-200, 200), (-1074, 1023)])
def test_reciprocal_roots(lib, ulps, lo, hi):
    """Significands and exponents (odd and even) over their ranges, powers of two and their neighbours, values that
    take the far routes and subnormal ones."""
    rng = np.random.default_rng(1000 + hi)
    n = 200000
    d = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))
    p = np.ldexp(1.0, np.arange(lo, hi))
    d = np.concatenate([d, p, np.nextafter(p, np.inf), np.nextafter(p, 0)[1:]])
    n = d.size
    fh, fl = np.empty(n, np.float32), np.empty(n, np.float32)
    r, s = np.empty(n), np.empty(n)
    lib.t_rsqrt(_ptr(d), n, ulps, _ptr(fh), _ptr(fl), _ptr(r), _ptr(s))
    root = np.sqrt(d.astype(np.longdouble))
    ok = (root > 2.0 ** -100) & (root < 2.0 ** 100)  # both parts of the pair inside FP32's normal range
    pair = fh[ok].astype(np.longdouble) + fl[ok].astype(np.longdouble)
    assert np.max(np.abs(pair * root[ok] - 1.0)) <= 2.0 ** -49 + 2.0 ** -52
    normal = d >= 2.0 ** -1022
    assert np.max(np.abs(r * root - 1.0)[normal]) <= 1.5 * 2.0 ** -53 + 2.0 ** -62
    assert np.max(np.abs(s / root - 1.0)[normal]) <= 2.0 ** -53 + 2.0 ** -62
    if not np.all(normal):  # FP64's own square root and division
        assert np.max(np.abs(r * root - 1.0)[~normal]) <= 2.0 ** -52 + 2.0 ** -62


def test_conversions(lib):
    """FP64 to a pair: hi is a nearest FP32 number (subnormal ones, where nothing is left for lo, ties to even), lo the
    nearest to what is left; and back.  Every exponent up to 2^126, significands at the edges of the rounding."""
    rng = np.random.default_rng(7)
    e = np.arange(-1074, 126)
    frac = np.concatenate([[1.0, 1.5, 2.0 - 2.0 ** -52], 1.0 + 2.0 ** -rng.integers(1, 53, 40).astype(float),
                           1.0 + 2.0 ** -24 + np.array([-1, 0, 1]) * 2.0 ** -52, 1.0 + 3 * 2.0 ** -24 + np.array([-1, 0, 1]) * 2.0 ** -52,
                           rng.uniform(1.0, 2.0, 200)])
    x = np.ldexp(frac[None, :], e[:, None]).ravel()
    x = np.concatenate([x, -x, [0.0, -0.0]])
    n = x.size
    hi, lo, back = np.empty(n, np.float32), np.empty(n, np.float32), np.empty(n)
    lib.t_pair(_ptr(x), n, _ptr(hi), _ptr(lo), _ptr(back))
    near = x.astype(np.float32).astype(np.float64)
    hi64 = hi.astype(np.float64)
    np.testing.assert_array_equal(np.abs(x - hi64), np.abs(x - near))  # a tie may go either way: lo makes it good
    tiny = np.abs(x) < 2.0 ** -126
    np.testing.assert_array_equal(hi64[tiny], near[tiny])
    np.testing.assert_array_equal(np.signbit(hi64), np.signbit(near))
    rest, lo64 = x - hi64, lo.astype(np.float64)
    sub = np.abs(rest) < 2.0 ** -126  # to 24 bits first, then to units of 2^-149: 3/4 of one
    np.testing.assert_array_equal(lo64[~sub], rest.astype(np.float32)[~sub])
    assert np.max(np.abs(rest - lo64)[sub]) <= 0.75 * 2.0 ** -149
    np.testing.assert_array_equal(back, hi64 + lo64)
