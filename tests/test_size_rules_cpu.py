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
    return lib


@pytest.mark.parametrize("S", [5, 6])
def test_wide_sums_begin_where_64_bits_end(rules, S):
    """k values add at most k 2^35 units of 2^-21, kept with 7 (S - 4) further bits in a signed 64-bit word: the
    limit is the smallest k (of 32-value steps) that may not fit, and no smaller one takes the slower conversion."""
    k = rules.wide_k(S)
    fits = lambda n: n * 2 ** 35 * 2 ** (7 * (S - 4)) < 2 ** 63
    assert fits(k - 32) and not fits(k)
