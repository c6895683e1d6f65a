"""Size rules of the tensor-core products (csrc/rules.h), compiled for the host."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09373_gb300", "csrc")

SOURCE = """
#include "rules.h"
extern "C" long long wide_k(int S) { return isdf::oz_wide_k(S); }
extern "C" int rule_splits(long long M, long long N, long long nkt, int S, int sym) {
  return isdf::oz_rule_splits(M, N, nkt, S, sym != 0);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    so = str(d / "librules.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "rules.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.wide_k.restype = ctypes.c_longlong
    lib.rule_splits.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 2
    return lib


@pytest.mark.parametrize("S", [5, 6])
def test_wide_sums_begin_where_64_bits_end(rules, S):
    """k values add at most k 2^35 units of 2^-21, kept with 7 (S - 4) further bits in a signed 64-bit word: the
    limit is the smallest k (of 32-value steps) that may not fit, and no smaller one takes the slower conversion."""
    k = rules.wide_k(S)
    fits = lambda n: n * 2 ** 35 * 2 ** (7 * (S - 4)) < 2 ** 63
    assert fits(k - 32) and not fits(k)


def test_splits_of_long_products(rules):
    """Partial results stay within 2 GiB however much a further split would help; the sizes the library is used at
    keep their splits; short products are left to the timing (0)."""
    assert rules.rule_splits(391, 208, 7, 8, 0) == 0
    assert rules.rule_splits(1657, 1657, 903168 // 32, 7, 1) == 16
    chosen = set()
    for n in (1000, 2500, 4100, 8000, 10000, 12000, 16400, 20000, 40000, 100000):
        for nkt in (1000, 30000, 400000):
            for S in (5, 6, 7, 8):
                for sym in (0, 1):
                    c = rules.rule_splits(n, n, nkt, S, sym)
                    assert c >= 1 and (c == 1 or 8 * c * n * n <= 2 ** 31), (n, nkt, S, sym, c)
                    chosen.add(c)
    assert len(chosen) > 1
