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
