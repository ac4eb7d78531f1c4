"""Krylov cycles on the N/2 and N/4 grids, against the oracle and against the plan's own grid alone.

Bars: the plan's usual ones (1e-10 mixed, 1e-12 FP64 at tol 1e-13, norm-wise), since the residual
on the plan's grid decides convergence whatever grid the cycles ran on.  Checked where the choice of
grid can go wrong: one and two coarse grids, slots that choose different grids in one batch, a
potential with modes that no coarse grid holds, a batch against single slots (value for value), graphs
on and off, small caps on cycles and iterations, and a memory budget without room for the grids.
"""
import numpy as np
import pytest

import workloads as wl
from oracle import dbar_oracle as orc

pytestmark = pytest.mark.gpu

L = 5.0


def rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / max(np.max(np.abs(np.asarray(b))), 1e-300))


@pytest.fixture(scope="module")
def dbar():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar as d
    return d


def smooth(N):
    return wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([1.4, 0.8 + 0.5j]))


def rough(N):
    """A disc with a jump: modes of every grid."""
    x = 2 * L * (np.arange(N) - N / 2) / N
    X, Y = np.meshgrid(x, x)
    return np.where((X - 0.4) ** 2 + Y ** 2 < 1.7, 1.2 - 0.4j, 0.0).astype(complex)


K = np.array([0.3 - 0.2j, -2.5j, 0.0])  # different shares of high modes: e_k moves the spectrum


@pytest.mark.parametrize("N", [256, 512])
@pytest.mark.parametrize("make", [smooth, rough])
@pytest.mark.parametrize("kw,bar", [(dict(prec="mixed", tol=1e-12), 1e-10),
                                    (dict(prec="mixed", resid_mode="fp64", sstep=2, tol=1e-12), 1e-10),
                                    (dict(prec="fp64", tol=1e-13), 1e-12)])
def test_coarse_cycles_match_oracle(dbar, N, make, kw, bar):
    Q = make(N)
    r = dbar.Plan(N, L, restart=16, max_batch=2, **kw).solve(Q, K, want_m=False)  # batches of 2 and 1
    one = dbar.Plan(N, L, restart=16, max_batch=1, graphs=0, **kw).solve(Q, K, want_m=False)
    assert r["status"] == dbar.DBAR_OK
    assert np.array_equal(r["S"], one["S"]) and np.array_equal(r["iters"], one["iters"])
    for i in range(K.size) if N == 256 else (1,):
        assert rel(r["S"][i], orc.solve_cgo(Q, K[i], N, L, tol=1e-14, restart=60)["S"]) < bar, i


def test_a_budget_without_room_for_the_grids_takes_the_plan_alone(dbar):
    N, Q = 512, smooth(512)
    kw = dict(prec="mixed", restart=16, tol=1e-12)
    full = dbar.Plan(N, L, max_batch=2, **kw)
    alone = dbar.Plan(N, L, max_batch=2, mem_budget=full.device_bytes - 1, **kw)
    assert alone.max_batch == 2 and alone.device_bytes < 0.9 * full.device_bytes
    a, f = alone.solve(Q, K[:2], want_m=False), full.solve(Q, K[:2], want_m=False)
    assert a["status"] == dbar.DBAR_OK and f["status"] == dbar.DBAR_OK
    assert rel(a["S"], f["S"]) < 2e-10  # each within 1e-10 of the solution
    with pytest.raises(dbar.DbarError) as e:
        dbar.Plan(N, L, max_batch=2, mem_budget=alone.device_bytes // 2, **kw)
    assert e.value.status == dbar.DBAR_ENOMEM


@pytest.mark.parametrize("caps", [dict(max_outer=1), dict(max_outer=3), dict(max_iter=16), dict(max_iter=24)])
def test_small_caps_leave_what_the_plan_alone_reaches(dbar, caps):
    # a cap that ends the solve early: the residual is at most that of a plan without coarse grids,
    # up to two blocks' progress, a decade each, where the cycles differ (a restart costs one)
    N, Q = 256, smooth(256)
    kw = dict(prec="mixed", restart=16, tol=1e-12, max_batch=1, **caps)
    full = dbar.Plan(N, L, **kw)
    alone = dbar.Plan(N, L, mem_budget=full.device_bytes - 1, **kw)
    a, f = alone.solve(Q, K[:1], want_m=False), full.solve(Q, K[:1], want_m=False)
    assert f["resid"][0] <= 100 * max(a["resid"][0], 1e-12)
    assert f["iters"][0][0] <= caps.get("max_iter", 99) + 4 and f["iters"][0][1] <= caps.get("max_outer", 99)


def test_server_slots_on_coarse_grids_match_the_plan(dbar):
    srv = dbar.Server(2 << 30, prec="mixed", tol=1e-12, max_batch=3)
    Qs = [smooth(256), rough(256), 0.5 * smooth(256), 1j * smooth(256)]
    tickets = [srv.submit(256, L, Q, K[i % 3]) for i, Q in enumerate(Qs)]
    for i, t in enumerate(tickets):
        o = orc.solve_cgo(Qs[i], K[i % 3], 256, L, tol=1e-14, restart=60)
        assert rel(srv.wait(t)["S"], o["S"]) < 1e-10, i
    srv.close()
