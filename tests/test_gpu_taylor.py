"""The FP32 Taylor coefficients: no row is rounded against another before its products.

Fields with one value per row, at p1 = 0: powers of two on the even rows below N/2, whose products
with the tables are exact, and values near 2^-24 on their mirror rows N - p2, which a sum of both rows in FP32
would lose.  The coefficients are linear in the field: those of both sets together are the sums of those
of each (products rounded alike, sums over rows in double-float: 2^-40), where such a sum is off by 2^-25.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 256, 1024])
def test_mirror_rows_are_not_rounded_together(N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    plan = dbar.Plan(N, 5.0, M=2, prec="mixed", max_batch=3, autotune=0)
    S = np.zeros((3, N, N), np.complex64)
    p = np.arange(2, N // 2, 2)
    S[0, p, 0] = 1.0
    S[1, N - p, 0] = 0.47 * 2.0 ** -23
    S[2] = S[0] + S[1]
    c = dbar.dbar_taylor(plan.handle, 3, torch.from_numpy(S).cuda(), 2, fp32=True)
    c1 = c[:, 1]
    assert abs(c1[0]) > 0 and abs(c1[1]) > 2.0 ** -26 * abs(c1[0])
    off = abs(c1[2] - c1[0] - c1[1]) / abs(c1[0])
    print(N, c1, off)
    assert off < 2.0 ** -40
