"""Algorithmic bytes of the profile: a potential that all slots share is read once per launch."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def test_shared_potential_counts_once():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    N, nb = 256, 8
    Q = wl.gaussian_mixture(N, 5.0, np.array([[0.3, -0.2]]), np.array([1.1]), np.array([1.4]))
    plan = dbar.Plan(N, 5.0, prec="mixed", tol=1e-12, max_batch=nb)

    def rhs_bytes(k):
        dbar.dbar_profile(plan.handle, True)
        plan.solve(Q, k, want_m=False)
        return dbar.profile_table(plan.handle)["rhs"][2]

    one, all_ = rhs_bytes(np.full(1, 0.3 - 0.2j)), rhs_bytes(np.full(nb, 0.3 - 0.2j))
    # per point and slot b, x: 16 bytes each, the basis's first vector and its low part: 8 each; Q: 16, once
    assert all_ / one == pytest.approx((nb * 48 + 16) / (48 + 16), rel=1e-12)
