"""The mixed-precision solve on the potential's box, against the oracle (1e-10, the mixed bar).

The Krylov vectors hold one value per point of the box of nonzero Q.  Checked where that can go
wrong: boxes off the centre, of odd height, touching the grid's edge, one point wide, the whole
grid; potentials of different extent on one plan (captured cycles follow the box); slots of a
server with different boxes.
"""
import numpy as np
import pytest

import workloads as wl
from oracle import dbar_oracle as orc

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / max(np.max(np.abs(np.asarray(b))), 1e-300))


@pytest.fixture(scope="module")
def dbar():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar as d
    return d


def cut(N, x0, x1, y0, y1, seed=3):
    """A smooth random potential, exactly zero outside [x0, x1) x [y0, y1)."""
    rng = np.random.default_rng(seed)
    Q = np.zeros((N, N), complex)
    h, w = y1 - y0, x1 - x0
    win = np.outer(np.sin(np.pi * (np.arange(h) + 0.5) / h) ** 2, np.sin(np.pi * (np.arange(w) + 0.5) / w) ** 2)
    Q[y0:y1, x0:x1] = win * (rng.uniform(0.5, 1.0) + 0.4j * rng.uniform(0.5, 1.0, (h, w)))
    return Q


BOXES = [(32, 2.0, (3, 20, 9, 30)), (64, 3.0, (0, 64, 0, 64)), (64, 3.0, (40, 64, 0, 13)), (128, 4.0, (60, 61, 70, 71)),
         (256, 6.0, (97, 160, 101, 152))]


@pytest.mark.parametrize("N,L,b", BOXES)
@pytest.mark.parametrize("M,sstep", [(0, 4), (2, 4), (7, 2), (2, 1)])
def test_box_solves_match_oracle(dbar, N, L, b, M, sstep):
    Q, k = cut(N, *b), np.array([0.3 - 0.2j, -0.7j, 0.0])
    plan = dbar.Plan(N, L, M=M, prec="mixed", restart=16, tol=1e-12, max_batch=2, sstep=sstep)  # batches of 2 and 1
    r = plan.solve(Q, k, want_m=False)
    assert r["status"] == dbar.DBAR_OK
    for i in range(k.size):
        o = orc.solve_cgo(Q, k[i], N, L, M=M, tol=1e-14, restart=60)
        assert rel(r["S"][i], o["S"]) < 1e-10, i


def test_potentials_of_different_extent_on_one_plan(dbar):
    # narrow, wide, narrow again, zero, with and without an initial guess: each solve is that
    # potential's own, whatever the plan solved before
    N, L, k = 128, 5.0, np.array([0.4 + 0.1j, -0.3j])
    plan = dbar.Plan(N, L, prec="mixed", restart=16, tol=1e-12, max_batch=2)
    narrow, wide = cut(N, 60, 72, 55, 66), wl.mixed_1024(N=N, nk=1, L=L).Q
    for Q in (narrow, wide, narrow):
        ref = [orc.solve_cgo(Q, kk, N, L, tol=1e-14, restart=60)["S"] for kk in k]
        r = plan.solve(Q, k, want_m=False)
        x = plan.solve(Q, k, want_m=False, x0=np.stack(ref) * 1.01)
        assert r["status"] == dbar.DBAR_OK and x["status"] == dbar.DBAR_OK
        for i in range(k.size):
            assert rel(r["S"][i], ref[i]) < 1e-10 and rel(x["S"][i], ref[i]) < 1e-10, i
    z = plan.solve(np.zeros((N, N)), k, want_m=False)
    assert z["status"] == dbar.DBAR_OK and np.all(z["S"] == 0)


def test_slots_with_different_boxes_match_oracle(dbar):
    N, L = 64, 3.0
    srv = dbar.Server(2 << 30, prec="mixed", tol=1e-12, max_batch=3)
    Qs = [cut(N, *b, seed=i) for i, b in enumerate([(0, 64, 0, 64), (30, 36, 20, 45), (1, 9, 50, 64), (31, 33, 31, 33)])]
    tickets = [srv.submit(N, L, Q, 0.2 - 0.1j * i) for i, Q in enumerate(Qs)]
    for i, t in enumerate(tickets):
        o = orc.solve_cgo(Qs[i], 0.2 - 0.1j * i, N, L, tol=1e-14, restart=60)
        assert rel(srv.wait(t)["S"], o["S"]) < 1e-10, i
    srv.close()


@pytest.mark.parametrize("N,L,b", BOXES)
@pytest.mark.parametrize("nk", [1, 40])
def test_fp64_box_solves_match_oracle(dbar, N, L, b, nk):
    # FP64 on the box; one slot (the small block shapes) and forty (the ordinary ones at N >= 64)
    Q = cut(N, *b)
    k = np.concatenate([[0.3 - 0.2j], 0.5 * np.exp(1j * np.arange(nk - 1))])
    plan = dbar.Plan(N, L, prec="fp64", restart=16, tol=1e-13, max_batch=nk)
    r = plan.solve(Q, k, want_m=False)
    assert r["status"] == dbar.DBAR_OK
    for i in (0, nk - 1):
        assert rel(r["S"][i], orc.solve_cgo(Q, k[i], N, L, tol=1e-14, restart=60)["S"]) < 1e-12, i


def test_entries_below_the_cut_change_nothing(dbar):
    # entries under 2^-100 of the largest are outside the box; the solution is the oracle's with them
    N, L = 64, 3.0
    Q = cut(N, 20, 44, 18, 40)
    far = Q + 1e-31 * np.abs(np.random.default_rng(2).standard_normal((N, N)))
    for prec, tol, bar in (("fp64", 1e-13, 1e-12), ("mixed", 1e-12, 1e-10)):
        r = dbar.Plan(N, L, prec=prec, restart=16, tol=tol, max_batch=1).solve(far, [0.4 - 0.3j])
        o = orc.solve_cgo(far, 0.4 - 0.3j, N, L, tol=1e-14, restart=60)
        assert r["status"] == dbar.DBAR_OK and rel(r["S"][0], o["S"]) < bar and rel(r["m"][0], o["m"]) < bar


@pytest.mark.parametrize("restart,sstep", [(100, 4), (128, 2)])
def test_long_cycles_match_oracle(dbar, restart, sstep):
    # the block scalar step's lane loops over more than 32 rows (106 to 147 iterations)
    N, L = 64, 3.0
    Q = 6.0 * cut(N, 2, 62, 2, 62)
    r = dbar.Plan(N, L, prec="fp64", restart=restart, sstep=sstep, tol=1e-13, max_batch=1).solve(Q, [0.9j])
    o = orc.solve_cgo(Q, 0.9j, N, L, tol=1e-14, restart=100)
    assert r["status"] == dbar.DBAR_OK and rel(r["S"][0], o["S"]) < 1e-11
