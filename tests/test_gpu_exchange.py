"""The tensor-core exchange at the edges of its blocks: pivot counts around the tiles of W (32) and of the products
(32 k, 48 and 128 rows), k ranges of [X^L X^N] that share a k tile, and levels without pivots or functions.

K and K C are compared with FP64 products of the library's own X^L, X^N and V.  Tolerance: every 5-digit product of
inner length k errs by at most u k max|a| max|b|, u = 2^-33, and carries its operands' errors on; the bounds of the
stages (Y, R, W, T or U, K or K C) are added up below.
"""
import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu
U = 2.0 ** -33


def _cell(levels):
    rng = np.random.default_rng(33)
    grids = ((16, 16, 16), (8, 8, 8), (4, 4, 4))[:levels]
    return S.make_system((1, 1, 1), 0.05, rng, grids, S.LEVEL_EDGES_3[: levels - 1]), rng


def _product(a, da, b, db):
    """a b^T and the bound of its error from those of a and b."""
    k = a.shape[1]
    ma, mb = np.abs(a).max(initial=0.0) + da, np.abs(b).max(initial=0.0) + db
    return a @ b.T, k * (ma * db + da * mb + U * ma * mb)


@pytest.mark.parametrize("levels,nip,drop", [(1, 1, None), (1, 31, None), (1, 33, None), (1, 161, None), (2, 96, None),
                                             (2, 129, 0), (3, 64, None), (3, 97, None), (3, 230, None), (3, 230, 0),
                                             (3, 230, 1), (3, 230, 2)])
@pytest.mark.parametrize("n", [1, 33])
def test_blocks_of_the_exchange(levels, nip, drop, n):
    sysd, rng = _cell(levels)
    N = S.nbasis(sysd)
    C = np.linalg.qr(rng.standard_normal((N, n)))[0].copy()
    plan = B.isdf_plan(sysd, {"precision": 1})
    try:
        piv, _ = B.isdf_select_points(plan, nip)
        if drop is not None:
            piv = piv[(piv >> B.PIVOT_SHIFT) != drop]
        B.isdf_fit(plan, piv)
        B.isdf_coulomb(plan)
        k = piv.size
        XL = B.isdf_get(plan, B.GET_XL).reshape(N, k)
        XN = B.isdf_get(plan, B.GET_XN).reshape(N, k)
        V = B.isdf_get(plan, B.GET_V).reshape(k, k)
        K, Ex = B.isdf_exchange(plan, C)
        KC, Exo = B.isdf_exchange_occ(plan, C)
        again, _ = B.isdf_exchange(plan, C)
    finally:
        plan.close()
    yl, e1 = _product(XL.T, 0.0, C.T, 0.0)
    yn, e2 = _product(XN.T, 0.0, C.T, 0.0)
    yg, eg = yl + yn, e1 + e2
    rgg, d1 = _product(yg, eg, yg, eg)
    rgl, d2 = _product(yg, eg, yl, e1)
    rll, d3 = _product(yl, e1, yl, e1)
    W = np.block([[V * rgg, V * rgl], [V * rgl.T, V * rll]])
    dW = np.abs(V).max() * max(d1, d2, d3)
    X2 = np.concatenate([XL, XN], axis=1)
    T, dT = _product(W, dW, X2, 0.0)
    want, dK = _product(X2, 0.0, T.T, dT)
    K, KC = np.asarray(K).reshape(N, N), np.asarray(KC).reshape(N, n)
    assert np.abs(K - want).max() <= dK
    assert np.array_equal(np.asarray(again).reshape(N, N), K)
    wc, dc = _product(want, dK, C.T, 0.0)
    y2 = np.concatenate([yl, yn])
    Uo, dU = _product(W, dW, y2.T, max(e1, e2))
    _, do = _product(X2, 0.0, Uo.T, dU)
    assert np.abs(KC - wc).max() <= do + 2.0 ** -50 * np.abs(wc).max()
    ex = -np.sum(C * wc)
    assert abs(Ex - ex) <= N * n * np.abs(C).max() * dc
    assert abs(Exo - ex) <= N * n * np.abs(C).max() * (do + 2.0 ** -50 * np.abs(wc).max())
