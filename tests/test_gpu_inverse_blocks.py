"""R^-1 of the tensor-core fit at the edges of its blocks (64-row diagonal blocks, doubling, products of halves of 256
rows and more on the tensor cores), through Xi = ZC^T (CC^T + lambda I)^-1 of isdf_fit: every grid point has its own
bound, so that a wrong block shows wherever its rows count.

Bound (precision 1), first order in the 5-digit products' errors.  A product of rows x and y over K values is off by at
most e K max|x| max|y|, e = 2^-31 (2^-33 and the powers of two above the maxima).  With S(p, g) = sum_r |phi_r(p) phi_r(g)|:
dZC = 2 S dA + dA^2, dA = e nfun max|phi(g)| max|phi(p)|; Y = R^-1 ZC is off by dY = e k max|ZC(:, g)| max|R^-1(j, :)|, Xi =
R^-T Y by dX = e k max|Y(:, g)| max|R^-1(:, j)|; so (CC^T + lambda I) Xi misses ZC by at most |R| dY + |A| dX + dZC + dCC |Xi|.
FP64 Cholesky and 8-digit products are below that.  The CPU test plants a wrong block in FP64 NumPy."""
import numpy as np
import pytest

import oracle.isdf as O
from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

REG = 1e-3  # lambda = REG tr(CC^T) / k
E5 = 2.0 ** -31


def _cell():
    return S.make_system((1, 1, 1), 0.05, np.random.default_rng(21), ((16, 18, 12),), ())


class Normal:
    """The normal equations of one level from its basis values, and the bound of their residual."""

    def __init__(self, phi, piv):
        P, k = phi[:, piv], len(piv)
        self.zc = (P.T @ phi) ** 2
        self.A = self.zc[:, piv] + REG * np.trace(self.zc[:, piv]) / k * np.eye(k)
        self.R = np.linalg.cholesky(self.A)
        self.Ri = np.tril(np.linalg.inv(self.R))
        y = self.Ri @ self.zc
        dA = E5 * phi.shape[0] * np.abs(phi).max(0)[None, :] * np.abs(P).max(0)[:, None]
        dZ = 2.0 * (np.abs(P).T @ np.abs(phi)) * dA + dA ** 2
        dY = E5 * k * np.abs(self.zc).max(0)[None, :] * np.abs(self.Ri).max(1)[:, None]
        dX = E5 * k * np.abs(y).max(0)[None, :] * np.abs(self.Ri).max(0)[:, None]
        dCC = dZ[:, piv] + REG * np.trace(dZ[:, piv]) / k * np.eye(k)
        self.bound = np.abs(self.R) @ dY + np.abs(self.A) @ dX + dZ + dCC @ np.abs(self.Ri.T @ y)

    def miss(self, xi):
        return np.abs(self.A @ xi - self.zc) / self.bound


@pytest.mark.gpu
@pytest.mark.parametrize("k", [1, 63, 64, 65, 128, 129, 257, 330, 511, 512, 513, 600, 769])
def test_tensor_core_fit_solves_its_normal_equations_at_every_point(k):
    plan = B.isdf_plan(_cell(), {"precision": 1, "reg_rel": REG})
    try:
        piv, _ = B.isdf_select_points(plan, k)
        B.isdf_fit(plan, piv)
        ng = int(np.prod(plan.system["grids"][0]))
        phi = B.isdf_get(plan, B.GET_PHI_LEVEL0).reshape(-1, ng)
        xi = B.isdf_get(plan, B.GET_XI_LEVEL0).reshape(k, ng)
    finally:
        plan.close()
    assert np.all(np.isfinite(xi))
    assert np.max(Normal(phi, piv).miss(xi)) <= 1.0


@pytest.mark.parametrize("k", [129, 600])
def test_the_bound_shows_a_wrong_block(k):
    sysd = _cell()
    lev = O._level_data(sysd, O.expand_functions(sysd))
    piv = np.asarray(O.select_points(lev, k)["pivots"])  # one level: the codes are the grid points
    eq = Normal(np.concatenate([lev[0]["PhiL"], lev[0]["PhiN"]]), piv)
    good = eq.Ri.T @ (eq.Ri @ eq.zc)
    assert np.max(eq.miss(good)) <= 1e-3
    h = 64 if k < 512 else 256
    for rows, cols in ((slice(h, k), slice(0, h)), (slice(64, 96), slice(0, 32)), (slice(k - 1, k), slice(0, 64))):
        Ri = eq.Ri.copy()
        Ri[rows, cols] = 0.0
        miss = eq.miss(Ri.T @ (Ri @ eq.zc))
        assert np.mean(miss.max(0) > 1.0) > 0.99  # at every grid point, or almost (part of the last row alone)
