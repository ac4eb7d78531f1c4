"""||b||, by which a solve's residual and stopping test are measured, to FP32 rounding of short sums.

In the double-float path squares are formed in FP32.  Here each thread of the right-hand side's
kernel meets one large value and then 255 whose squares are 2^-25.1 of its square: sums held in FP32
over all of them lose every one (3.5e-6 of the norm).  Bound: 14 roundings of 2^-24 in ||b||^2 (conversion,
squares, sums of at most 8 values), 24 in ||r||^2 (sums of 16 and across lanes), half of each in the norms,
1.2e-6 together, rounded up to 1.5e-6.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_reported_residual_of_a_wide_potential():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    N, L, k = 2048, 5.0, np.array([0.3 - 0.2j])
    Q = np.full((N, N), 0.25 * 2.0 ** -12.55, complex)
    Q[:64, :256] = 0.25
    plan = dbar.Plan(N, L, prec="mixed", restart=4, inner_tol=1e-3, tol=1e-4, max_outer=1, max_batch=1)
    r = plan.solve(Q, k, want_m=False)
    got = r["resid"][0]
    assert 1e-8 < got < 1e-1
    exact = dbar.Plan(N, L, prec="fp64", restart=4, max_batch=1)
    Qd, S = torch.from_numpy(Q).cuda(), torch.from_numpy(r["S"]).cuda()
    AS, b = torch.empty_like(S), torch.empty_like(S)
    dbar.dbar_apply(exact.handle, Qd, k, S, AS)
    dbar.dbar_rhs(exact.handle, Qd, k, b)
    want = float(torch.linalg.norm(b - AS) / torch.linalg.norm(b))
    print(f"resid {got:.9e}, in FP64 {want:.9e}, off by {got / want - 1:.2e}")
    assert abs(got / want - 1) < 1.5e-6
