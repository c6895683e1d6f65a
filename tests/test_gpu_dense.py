"""Cholesky of CC^T and the inverse of its factor at the edges of their blocks (64-row block columns, 32 x 32
tiles, doubling of the inverted blocks), through isdf_fit: Xi CC^T = ZC^T with M_l built from the library's own
basis values.

Tolerance: Xi = (ZC^T R^-T) R^-1 with an explicit inverse carries a relative error of about k eps in each
product with R^-1, and multiplying back by CC^T = R R^T leaves k eps |R^-1| |R| = k eps sqrt(cond) of ZC^T; 8
times that is allowed.
"""
import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _cell():
    rng = np.random.default_rng(21)
    return S.make_system((1, 1, 1), 0.05, rng, ((16, 18, 12),), ())


@pytest.mark.parametrize("k", [1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 129, 191, 257, 330])
@pytest.mark.parametrize("precision", [0, 1])
def test_fit_solves_its_normal_equations(k, precision):
    sysd = _cell()
    plan = B.isdf_plan(sysd, {"precision": precision})
    try:
        piv, _ = B.isdf_select_points(plan, k)
        B.isdf_fit(plan, piv)
        ng = int(np.prod(sysd["grids"][0]))
        phi = B.isdf_get(plan, B.GET_PHI_LEVEL0).reshape(-1, ng)
        xi = B.isdf_get(plan, B.GET_XI_LEVEL0).reshape(k, ng)
    finally:
        plan.close()
    zc = (phi[:, piv].T @ phi) ** 2
    cc = zc[:, piv]
    back = cc @ xi
    eps = 2.0 ** -52 if precision == 0 else 2.0 ** -33 * phi.shape[0]  # 5-digit products form ZC^T and Xi
    tol = 8.0 * k * eps * np.sqrt(np.linalg.cond(cc)) * np.abs(zc).max()
    assert np.all(np.isfinite(xi))
    assert np.abs(back - zc).max() <= tol


def test_several_levels_factor_together():
    """Levels of very different size (and one without pivots) go through the same launches."""
    rng = np.random.default_rng(5)
    sysd = S.make_system((1, 1, 1), 0.05, rng, ((16, 16, 16), (8, 8, 8), (4, 4, 4)), S.LEVEL_EDGES_3)
    plan = B.isdf_plan(sysd)
    try:
        piv, _ = B.isdf_select_points(plan, 230)
        lev = piv >> B.PIVOT_SHIFT
        for sets in (piv, piv[lev != 1], np.concatenate([piv[lev == 0][:70], piv[lev == 2][:3]])):
            B.isdf_fit(plan, sets)
            V = np.zeros((sets.size, sets.size))
            B.isdf_coulomb(plan, V)
            lo = np.concatenate([sets[(sets >> B.PIVOT_SHIFT) == l] for l in range(3)])
            for l in range(3):
                g = lo[(lo >> B.PIVOT_SHIFT) == l] & ((1 << B.PIVOT_SHIFT) - 1)
                if not g.size:
                    continue
                ng = int(np.prod(sysd["grids"][l]))
                phi = B.isdf_get(plan, B.GET_PHI_LEVEL0 + l).reshape(-1, ng)
                xi = B.isdf_get(plan, B.GET_XI_LEVEL0 + l).reshape(g.size, ng)
                nL = (5, 4, 4)[l] * 8
                aL, aN = phi[:nL, g].T @ phi[:nL], phi[nL:, g].T @ phi[nL:]
                zc = aL * (aL + 2.0 * aN)
                cc = zc[:, g]
                tol = 8.0 * g.size * 2.0 ** -52 * np.sqrt(np.linalg.cond(cc)) * np.abs(zc).max()
                assert np.abs(cc @ xi - zc).max() <= tol
            assert np.all(np.isfinite(V)) and np.array_equal(V, V.T)
    finally:
        plan.close()
