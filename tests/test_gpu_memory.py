"""Device memory of plans and servers with coarse grids.

A level's Krylov basis lies in the plan's own basis, so the grids add the levels' fields and tables only.
Per slot in units of N^2 elements (mixed precision, restart m): the plan holds 4 fields of 16 bytes and m + 2 of 8,
the levels (1/4 + 1/16) of 4 fields of 16 bytes and one of 8; tables the same share of the plan's.
"""
import gc

import numpy as np
import pytest

import workloads as wl
from oracle import dbar_oracle as orc

pytestmark = pytest.mark.gpu

L = 5.0


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    return torch, dbar


def smooth(N):
    return wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([1.4, 0.8 + 0.5j]))


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("prec,elem", [("mixed", 8), ("fp64", 16)])
def test_levels_share_the_basis(gpu, prec, elem):
    torch, dbar = gpu
    N, m = 512, 32
    kw = dict(prec=prec, restart=m, tol=1e-12)
    size = {nb: dbar.Plan(N, L, max_batch=nb, **kw).device_bytes for nb in (4, 8)}
    per_slot = (size[8] - size[4]) / 4
    alone = N * N * (64 + (m + 2) * elem)
    levels = N * N * 5 / 16 * (64 + elem)
    assert per_slot < 1.02 * (alone + levels)  # (a basis per level: 1.17 to 1.2 times that)


@pytest.mark.parametrize("prec,tol,bar", [("mixed", 1e-12, 1e-10), ("fp64", 1e-13, 1e-12)])
def test_slots_on_every_grid_at_once(gpu, prec, tol, bar):
    # smooth and oscillating right-hand sides: slots of one batch iterate on different grids at the same time
    torch, dbar = gpu
    N = 512
    k = np.array([0.1, -2.5j, 0.0, 9.0 - 8.0j, 0.3 - 0.2j, 14.0, 0.5j, 4.0 + 1.0j])
    plan = dbar.Plan(N, L, prec=prec, restart=16, tol=tol, max_batch=8)
    for _ in range(3):
        r = plan.solve(smooth(N), k, want_m=False)
        assert r["status"] == dbar.DBAR_OK
    one = dbar.Plan(N, L, prec=prec, restart=16, tol=tol, max_batch=1)
    for i in range(k.size):
        assert np.array_equal(r["S"][i], one.solve(smooth(N), k[i:i + 1], want_m=False)["S"][0]), i
    for i in (1, 3):
        assert rel(r["S"][i], orc.solve_cgo(smooth(N), k[i], N, L, tol=1e-14, restart=60)["S"]) < bar, i


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_the_automatic_batch_is_what_fits_without_coarse_grids(gpu, prec):
    # dbar_apply and its kind take at most max_batch fields: room for the grids must not lower it
    torch, dbar = gpu
    N, kw = 256, dict(prec=prec, restart=16, tol=1e-12)
    full = dbar.Plan(N, L, max_batch=7, **kw).device_bytes
    alone = dbar.Plan(N, L, max_batch=7, mem_budget=full - 1, **kw).device_bytes  # without them
    assert alone < full
    tight = dbar.Plan(N, L, max_batch=0, mem_budget=alone, **kw)
    assert tight.max_batch == 7 and tight.device_bytes == alone
    roomy = dbar.Plan(N, L, max_batch=0, mem_budget=full, **kw)
    assert roomy.max_batch >= 7 and roomy.device_bytes <= full
    assert tight.solve(smooth(N), [0.3 - 0.2j], want_m=False)["status"] == dbar.DBAR_OK


def test_a_lane_without_room_for_its_grids_leaves_idle_lanes_alone(gpu):
    # a budget for both grid classes, the larger one without coarse grids (they take a sixth of it): the idle
    # lane of the smaller class keeps its plan, and its next request finds it
    torch, dbar = gpu

    def held():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    n, S, m = 1024 * 1024, 4, 32
    slot = n * (4 * 16 + (m + 2) * 8 + 40) + ((m + 1) * S + 10) * 128 * 8 + (S * (S + m + 1) + m * (m + 1)) * 8
    alone = slot + 13 * 16 * n  # a one-slot lane of 1024^2 by the server's own estimate, and the grids beyond it
    grids = n * 5 // 16 * (4 * 16 + 8 + 40) + 13 * 16 * n * 5 // 16
    kw = dict(prec="mixed", tol=1e-12, max_batch=1)
    Qa, Qb, k = smooth(512), smooth(1024), 0.3 - 0.2j
    gc.collect()  # plans of earlier tests
    before = held()
    srv = dbar.Server(8 << 30, **kw)
    srv.wait(srv.submit(512, L, Qa, k))
    small = before - held()
    srv.close()
    srv = dbar.Server(small + alone + grids // 2, **kw)
    assert srv.wait(srv.submit(512, L, Qa, k))["status"] == dbar.DBAR_OK
    assert srv.wait(srv.submit(1024, L, Qb, k))["status"] == dbar.DBAR_OK
    both = held()
    got = srv.wait(srv.submit(512, L, Qa, k))
    assert got["status"] == dbar.DBAR_OK
    assert abs(held() - both) < 32 << 20 and before - both > small + 0.8 * alone
    assert rel(got["S"], orc.solve_cgo(Qa, k, 512, L, tol=1e-14, restart=60)["S"]) < 1e-10
    srv.close()
