"""Caps on iterations and cycles: what the plan's own grid reaches within them, a plan with coarse grids reaches too.

Solves that end just within their cap on the plan's own grid (a plan whose memory leaves no room for coarse
grids); with iterations and cycles on coarse grids counted against the caps each of these missed tol.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

L = 5.0


def mixture(N, a):
    return a * wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([1.4, 0.8 + 0.5j]))


def disc(N):
    x = 2 * L * (np.arange(N) - N / 2) / N
    X, Y = np.meshgrid(x, x)
    return np.where((X - 0.4) ** 2 + Y ** 2 < 1.7, 1.2 - 0.4j, 0.0).astype(complex)


K = np.concatenate([[0.1, 0.3 - 0.2j, -2.5j, 0.0], 8 * np.exp(1j * np.arange(4)), 20 * np.exp(0.7j * np.arange(4))])
CASES = [(256, "mixed", 32, 3.0, dict(max_iter=48)), (256, "fp64", 32, 1.0, dict(max_iter=20)),
         (256, "fp64", 32, 3.0, dict(max_iter=40)), (256, "fp64", 32, 3.0, dict(max_iter=48)),
         (512, "fp64", 16, 1.0, dict(max_iter=16)), (512, "fp64", 32, 1.0, dict(max_iter=24)),
         (256, "fp64", 16, 0.0, dict(max_outer=4)), (512, "fp64", 16, 0.0, dict(max_iter=40)),
         (256, "fp64", 8, 3.0, dict(max_iter=64)), (512, "mixed", 8, 3.0, dict(max_iter=64, max_outer=8)),
         (512, "fp64", 4, 3.0, dict(max_iter=64, max_outer=16))]


@pytest.mark.parametrize("N,prec,restart,a,caps", CASES)
def test_caps_hold_for_the_plans_own_grid(N, prec, restart, a, caps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    Q = mixture(N, a) if a else disc(N)  # (a = 0: a potential with a jump)
    kw = dict(prec=prec, restart=restart, tol=1e-12 if prec == "mixed" else 1e-13, max_batch=K.size, autotune=0, **caps)
    full = dbar.Plan(N, L, **kw)
    alone = dbar.Plan(N, L, mem_budget=full.device_bytes - 1, **kw)
    f, o = full.solve(Q, K, want_m=False), alone.solve(Q, K, want_m=False)
    ended = o["resid"] <= kw["tol"]
    assert np.all(f["resid"][ended] <= kw["tol"]), (o["iters"][ended].tolist(), f["iters"][ended].tolist())
    most = np.array([1.5 * kw.get("max_iter", 4000), 1.5 * kw.get("max_outer", 40)])
    assert np.all(f["iters"] <= most + [4, 0])
