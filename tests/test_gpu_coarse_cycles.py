"""Which grids the Krylov cycles ran on, and what one coarse cycle gains.

The true residual decides convergence whatever grid a cycle took, so right solutions alone do not show that
a coarse cycle ran, or that it gained anything.  From the profile's launches of the residual's passes: a
cycle's end takes one row, one column and one last pass, a correction from a coarse grid two row passes and one of
each, so corrections (one per part of a cycle and grid) = row passes - last passes.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

L = 5.0


@pytest.fixture(scope="module")
def dbar():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar as d
    return d


def smooth(N):
    return wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([1.4, 0.8 + 0.5j]))


def jump(N):
    x = 2 * L * (np.arange(N) - N / 2) / N
    X, Y = np.meshgrid(x, x)
    return np.where((X - 0.4) ** 2 + Y ** 2 < 1.7, 1.2 - 0.4j, 0.0).astype(complex)


def corrections(dbar, plan, Q, k):
    dbar.dbar_profile(plan.handle, True)
    r = plan.solve(Q, np.array(k), want_m=False)
    t = dbar.profile_table(plan.handle)
    return t["fp64_residual_pass_a"][1] - t["fp64_residual_pass_c"][1], r


@pytest.mark.parametrize("N", [512, 1024])
def test_smooth_residuals_never_see_the_fine_grid(dbar, N):
    plan = dbar.Plan(N, L, prec="mixed", restart=32, tol=1e-12, max_batch=1)
    n, r = corrections(dbar, plan, smooth(N), [0.3 - 0.2j])
    assert r["status"] == dbar.DBAR_OK and n == r["iters"][0][1] > 0  # every cycle on a coarse grid


def test_one_coarse_cycle_gains_what_it_aims_at(dbar):
    # FP64, a right-hand side that the N/4 or N/2 grid resolves to rounding: one coarse cycle, 13 decades
    N = 1024
    plan = dbar.Plan(N, L, prec="fp64", restart=32, tol=1e-13, max_batch=1)
    n, r = corrections(dbar, plan, smooth(N), [0.3 - 0.2j])
    assert n == 1 and r["iters"][0][1] == 1 and r["resid"][0] < 1e-13


@pytest.mark.parametrize("N", [256, 512])
def test_a_jump_stays_on_the_plans_grid(dbar, N):
    plan = dbar.Plan(N, L, prec="mixed", restart=32, tol=1e-12, max_batch=1)
    n, r = corrections(dbar, plan, jump(N), [0.3 - 0.2j])
    assert r["status"] == dbar.DBAR_OK and n == 0


def test_slots_of_one_batch_take_different_grids(dbar):
    N = 512
    plan = dbar.Plan(N, L, prec="mixed", restart=32, tol=1e-12, max_batch=2)
    low, _ = corrections(dbar, plan, smooth(N), [0.3 - 0.2j])
    high, h = corrections(dbar, plan, smooth(N), [20.0])
    both, b = corrections(dbar, plan, smooth(N), [0.3 - 0.2j, 20.0])
    assert low > 0 and high == 0 and both == low
    assert b["status"] == dbar.DBAR_OK and np.array_equal(b["S"][1], h["S"][0])
