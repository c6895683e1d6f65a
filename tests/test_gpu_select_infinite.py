"""Residuals that overflow: with every pair density of the sharpest functions above the range of a double no residual
can be compared, and the selection ends without points, step by step and in blocks alike."""
import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [0, 16, 96, 200])
@pytest.mark.parametrize("prefilter", [0, 1])
def test_infinite_residuals_end_the_selection(block, prefilter):
    # phi at its own centre is (2 alpha / pi)^(3/4), about 1e82; atoms sit on grid points
    sysd = S.make_system((1, 1, 1), 0.0, None, ((16, 16, 16),), (), s_exps=(0.1, 0.4, 1.6, 1e110))
    plan = B.isdf_plan(sysd, {"precision": 1, "select_block": block, "prefilter": prefilter})
    try:
        phi = B.isdf_get(plan, B.GET_PHI_LEVEL0)
        assert np.all(np.isfinite(phi)) and np.max(phi) > 1e80
        piv, val = B.isdf_select_points(plan, 40)
        assert len(piv) == 0 and len(val) == 0
    finally:
        plan.close()
