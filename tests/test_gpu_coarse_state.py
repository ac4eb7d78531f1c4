"""The choice of a cycle's grid where its inputs are no ordinary numbers.

Slots that never began (a lane opens more slots than it has requests) hold no state in memory that
other programs have used before, and an FP64 right-hand side far below FP32's range, whose shares of
modes are no numbers in FP32, takes the plan's own grid.
"""
import numpy as np
import pytest

import workloads as wl
from oracle import dbar_oracle as orc

pytestmark = pytest.mark.gpu

N, L = 256, 5.0


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    return torch, dbar


def smooth():
    return wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([1.4, 0.8 + 0.5j]))


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("scale", [1e-30, 1e-45, 1e-60])
def test_fp64_right_hand_sides_below_fp32(gpu, scale):
    # S is linear in so small a potential: the right-hand side itself, to far below 1e-12
    torch, dbar = gpu
    k = np.array([0.3 - 0.2j, -0.5j])
    plan = dbar.Plan(N, L, prec="fp64", restart=16, tol=1e-13, max_batch=2)
    r = plan.solve(scale * smooth(), k, want_m=False)
    assert r["status"] == dbar.DBAR_OK
    for i in range(2):
        assert rel(r["S"][i] / scale, orc.solve_cgo(1e-20 * smooth(), k[i], N, L, tol=1e-14)["S"] / 1e-20) < 1e-12


@pytest.mark.parametrize("prec,bar", [("mixed", 1e-10), ("fp64", 1e-12)])
def test_slots_that_never_begin(gpu, prec, bar):
    torch, dbar = gpu
    for byte in (0x01, 0x7f):  # memory another program left, in which the lane's state then lies
        t = torch.full((4 << 30,), byte, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        del t
        torch.cuda.empty_cache()
        srv = dbar.Server(3 << 30, prec=prec, tol=1e-12 if prec == "mixed" else 1e-13)
        k = np.array([0.3 - 0.2j, -2.5j])
        tickets = [srv.submit(N, L, smooth(), kk) for kk in k]  # two requests, at least nine slots
        for i, t in enumerate(tickets):
            got = srv.wait(t)
            assert got["status"] == dbar.DBAR_OK
            assert rel(got["S"], orc.solve_cgo(smooth(), k[i], N, L, tol=1e-14, restart=60)["S"]) < bar
        srv.close()
