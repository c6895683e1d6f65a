"""The product's integer sums at their limits: operands that are constant along k make the middle digit levels of a
chunk as large as digits allow (0.996: 19,281,920 in level 2 of a 1024-k chunk, beyond 2^24), and many k values make
the whole sum so (5 digits from 2^21 values on, 6 from 2^14, it leaves 64 bits before the scale and takes another
conversion).

Bound, from the digits alone: with |x| < X = 2^e of its row, rounding to 7 S bits leaves 2^-(7 S + 1) X an operand,
and the dropped digit pairs (s + t >= S, digits at most 64 there) (S - 1) 64^2 2^-(14 + 7 S) and 1/127 of that below;
in all K X Y 2^-(7 S) (1 + 0.252 (S - 1)), and 2^-53 |C| for the last rounding (2 splits - 1 of them with split k).
Rows constant along k add even
integers below 2^25 to every level, so FP32 accumulation is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(x, y, K, slices, splits=1):
    """C of rows constant along k: C[m][n] = K x_m y_n, in extended precision."""
    import torch

    from paper_2404_09373_gb300 import isdf as B

    a = torch.from_numpy(x).cuda()[:, None].expand(-1, K).contiguous()
    b = torch.from_numpy(y).cuda()[:, None].expand(-1, K).contiguous()
    c = torch.full((x.size, y.size), float("nan"), dtype=torch.float64, device="cuda")
    B.isdf_gemm_f64(a, b, c, slices=slices, splits=splits)
    C = c.cpu().numpy()
    xy = x.astype(np.longdouble)[:, None] * y.astype(np.longdouble)[None, :] * K
    scale = np.ldexp(1.0, np.frexp(x)[1])[:, None] * np.ldexp(1.0, np.frexp(y)[1])[None, :]
    bound = K * scale * 2.0 ** (-7 * slices) * (1.0 + 0.252 * (slices - 1)) + (2 * splits - 1) * 2.0 ** -53 * np.abs(xy)
    err = np.abs(C - xy)
    assert np.all(err <= bound), (int(np.sum(~(err <= bound))), float(np.max(err / np.abs(xy))))


@pytest.mark.parametrize("slices", [5, 6, 7, 8])
@pytest.mark.parametrize("K,splits", [(820, 1), (1024, 1), (1025, 1), (2048, 2), (3000, 1), (5000, 3)])
def test_rows_constant_along_k(slices, K, splits):
    rng = np.random.default_rng(K)
    x, y = rng.uniform(0.5, 1.0, 390), rng.uniform(0.5, 1.0, 290)
    x[:3], y[:3] = (0.996, -0.996, 1.0 - 2.0 ** -53), (0.996, -0.996, 1.0 - 2.0 ** -53)
    x[3::2] *= -1.0
    _check(x * np.exp2(rng.integers(-30, 30, size=x.size)), y, K, slices, splits)


@pytest.mark.parametrize("slices,K", [(5, 2 ** 21 - 1), (5, 2 ** 21), (5, 2 ** 21 + 33), (6, 2 ** 14 - 32), (6, 2 ** 14),
                                      (6, 2 ** 14 + 1), (7, 2 ** 14), (8, 2 ** 14)])
def test_sums_at_the_64_bit_limit(slices, K):
    x = np.array([0.996, -0.996, 1.0 - 2.0 ** -53, 0.75, 2.0 ** -300, -1e200, 0.5])
    y = np.array([0.996, 1.0 - 2.0 ** -53, -0.5, 0.999])
    _check(x, y, K, slices)
