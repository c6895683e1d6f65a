"""An expired wait ends a product as a whole: every warp of a CTA leaves together whichever of its lanes saw the
error first, with several tiles a CTA, ragged edges, split k, and in the selection's column kernel.  The waits are
made to expire from the host (ISDF_FAULT=oz_wait: a zero limit); the call reports ISDF_ERR_TIMEOUT and the same call
afterwards gives the bits it gave before."""
import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slices", [5, 6, 7, 8])
@pytest.mark.parametrize("M,N,K,splits", [(1024, 481, 2100, 1), (300, 97, 1500, 3), (40000, 96, 512, 1)])
def test_product_ends_and_recovers(monkeypatch, slices, M, N, K, splits):
    import torch

    g = torch.Generator(device="cuda").manual_seed(M + N)
    a = torch.randn((M, K), dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn((N, K), dtype=torch.float64, device="cuda", generator=g)
    c = torch.empty((M, N), dtype=torch.float64, device="cuda")
    want = B.isdf_gemm_f64(a, b, c, slices=slices, splits=splits).clone()
    monkeypatch.setenv("ISDF_FAULT", "oz_wait")
    for _ in range(3):
        with pytest.raises(B.IsdfError) as e:
            B.isdf_gemm_f64(a, b, c, slices=slices, splits=splits)
        assert e.value.status == B.ISDF_ERR_TIMEOUT
    monkeypatch.delenv("ISDF_FAULT")
    c.fill_(float("nan"))
    assert torch.equal(B.isdf_gemm_f64(a, b, c, slices=slices, splits=splits), want)


def test_selection_columns_end_and_recover(monkeypatch):
    rng = np.random.default_rng(8)
    sysd = S.make_system((1, 1, 1), 0.05, rng, ((24, 24, 24), (12, 12, 12), (6, 6, 6)), S.LEVEL_EDGES_3)
    plan = B.isdf_plan(sysd, {"precision": 1, "prefilter": 1, "select_block": 96})
    try:
        want, wval = B.isdf_select_points(plan, 200)
        monkeypatch.setenv("ISDF_FAULT", "oz_wait")
        with pytest.raises(B.IsdfError) as e:
            B.isdf_select_points(plan, 200)
        assert e.value.status == B.ISDF_ERR_TIMEOUT
        monkeypatch.delenv("ISDF_FAULT")
        piv, val = B.isdf_select_points(plan, 200)
        assert np.array_equal(piv, want) and np.array_equal(val, wval)
    finally:
        plan.close()
