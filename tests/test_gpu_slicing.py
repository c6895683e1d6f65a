"""Digit planes of the tensor-core operands, seen through isdf_gemm_f64 with B = the identity.

C[m, n] = A[m, n] then, up to the rounding of A's row to 7 S fraction bits of its scale: S digits hold
x 2^-e_r to 2^-(7 S + 1), and with 8 digits (56 bits below a power of two above the row's maximum) every
value within 2^3 of it exactly.  Shapes take each route of the row scales and digits: K below one k tile,
at its edges, one and several groups per warp, the last K of the one-pass kernel and the first beyond it,
ragged rows, and rows that are not 16-byte aligned.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slices", [5, 6, 7, 8])
@pytest.mark.parametrize("M,K,pad", [(1, 1, 0), (7, 31, 0), (129, 33, 1), (300, 255, 0), (300, 257, 3), (70, 513, 0),
                                     (9, 4096, 0), (9, 4097, 1), (5, 20000, 0)])
def test_rows_are_rounded_to_their_scale(M, K, pad, slices):
    import torch

    from paper_2404_09373_gb300 import isdf as B

    rng = np.random.default_rng(M + 7 * K + slices)
    A = rng.standard_normal((M, K)) * np.exp2(rng.integers(-200, 200, size=(M, 1)))
    A[:, ::5] *= 2.0 ** -20
    A[:, 3::11] = 0.0
    if M > 5:
        A[5] = 0.0
        A[6] = np.ldexp(1.0, -3) * np.sign(A[6])  # a row of equal magnitudes, a power of two
    n = min(K, 70)
    cols = rng.choice(K, size=n, replace=False)
    P = np.zeros((n, K))
    P[np.arange(n), cols] = 1.0
    buf = torch.zeros((M, K + pad), dtype=torch.float64, device="cuda")
    buf[:, :K] = torch.from_numpy(A)
    p = torch.from_numpy(P).cuda()
    c = torch.full((M, n), float("nan"), dtype=torch.float64, device="cuda")
    B.isdf_gemm_f64(buf[:, :K], p, c, slices=slices)
    got, want = c.cpu().numpy(), A[:, cols]
    top = np.abs(A).max(axis=1)
    e = np.where(top > 0, np.floor(np.log2(np.where(top > 0, top, 1.0))) + 1, 0)
    unit = np.exp2(e - 7 * slices)[:, None]
    # the products with B's single digit 64 2^-7 are exact; digits below the kept levels are dropped:
    # d_s with s = S - 1 .. stays (level s), so only A's own rounding is left, half a unit
    assert np.all(np.abs(got - want) <= 0.5 * unit + 2.0 ** -53 * np.abs(want))
    assert np.all(got[top == 0] == 0.0)
