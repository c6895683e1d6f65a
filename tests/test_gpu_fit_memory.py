"""Device memory at the height of the plain FP64 fit: the interpolation vectors of every level, and scratch of the
same size for one level at a time."""
import ctypes

import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


def _pool():
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool = ctypes.c_int(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0

    def get(attr):
        v = ctypes.c_uint64()
        assert cu.cuMemPoolGetAttribute(pool, attr, ctypes.byref(v)) == 0
        return v.value

    def reset():
        v = ctypes.c_uint64(0)
        assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, ctypes.byref(v)) == 0

    return get, reset


def test_fp64_fit_holds_scratch_of_one_level():
    import torch

    sysd = S.make_system((1, 1, 1), 0.05, np.random.default_rng(4), ((48, 48, 48), (46, 46, 46), (40, 40, 40)),
                         S.LEVEL_EDGES_3)
    ng = [int(np.prod(g)) for g in sysd["grids"]]
    plan = B.isdf_plan(sysd, {"precision": 0})
    try:
        piv, _ = B.isdf_select_points(plan, 400)
        lev = piv >> B.PIVOT_SHIFT
        piv = np.concatenate([piv[lev == l][:40] for l in range(3)])
        k = [int(np.sum((piv >> B.PIVOT_SHIFT) == l)) for l in range(3)]
        assert min(k) >= 30
        get, reset = _pool()
        torch.cuda.synchronize()
        reset()
        before = get(USED_CURRENT)
        B.isdf_fit(plan, piv)
        torch.cuda.synchronize()
        peak = get(USED_HIGH) - before
        vectors = [8 * a * b for a, b in zip(k, ng)]
        # the basis values at the pivots, k x k matrices, the factors X^L and X^N, residuals: below 16 MB here
        assert peak <= sum(vectors) + max(vectors) + 16 * 2 ** 20, (peak, vectors)
    finally:
        plan.close()
