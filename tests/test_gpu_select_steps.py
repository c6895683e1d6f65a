"""Ordinary selection steps (no speculative block) against pivoted Cholesky in NumPy on the library's own basis
values: candidate counts at the edges of a block's 256 values and a group's 32, one block and several, more pivots
asked than the matrix has, and selections that follow one another on a plan.

Tolerance of a pivot value after k steps: every step rounds a residual of at most d0 a few times, 16 k 2^-53 d0.
The pivots themselves have to be the same (the cell is displaced, and the tie rule is the library's)."""
import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu


def _greedy(M, nip, tie_rel, tie_abs):
    d = np.diag(M).copy()
    L = np.zeros((M.shape[0], nip))
    piv, val = [], []
    d0 = d.max()
    for k in range(nip):
        dmax = d.max()
        if not dmax > 1e-9 * d0:  # compared only where rounding does not decide
            break
        p = int(np.argmax(d >= dmax - max(tie_rel * dmax, tie_abs * d0)))
        piv.append(p)
        val.append(d[p])
        col = (M[:, p] - L[:, :k] @ L[p, :k]) / np.sqrt(d[p])
        col[p] = np.sqrt(d[p])
        L[:, k] = col
        d -= col * col
        d[p] = 0.0
    return np.array(piv), np.array(val), d0


@pytest.mark.parametrize("ncand", [1, 31, 33, 255, 256, 257, 513, 1728])
def test_steps_are_greedy(ncand):
    rng = np.random.default_rng(50)
    sysd = S.make_system((1, 1, 1), 0.05, rng, ((12, 12, 12),), ())
    ng = 1728
    cand = np.sort(rng.choice(ng, size=ncand, replace=False)).astype(np.int64)
    opts = B.default_options()
    plan = B.isdf_plan(sysd, {"precision": 0})
    try:
        phi = B.isdf_get(plan, B.GET_PHI_LEVEL0).reshape(-1, ng)[:, cand]
        w = np.prod(sysd["edges"]) / ng
        M = w * (phi.T @ phi) ** 2
        for nip in (min(ncand, 3), min(ncand, 90)):
            want, val, d0 = _greedy(M, nip, opts.tie_rel, opts.tie_abs)
            piv, dval = B.isdf_select_points(plan, nip, cand=cand)
            n = want.size
            assert np.array_equal(np.asarray(piv)[:n], cand[want])
            assert np.all(np.abs(np.asarray(dval)[:n] / dval[0] - val / val[0]) * val[0] <= 16 * n * 2.0 ** -53 * d0)
    finally:
        plan.close()
