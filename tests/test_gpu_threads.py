"""Host threads that solve on plans of their own at the same time.

Kernels that opt in to more than 48 KB of shared memory are shared by all plans of the process; a
launch's size depends on the basis size (block dots) and on the Taylor order (column passes).
Threads with graphs off launch every kernel directly, at restarts and orders of their own; each
solve returns DBAR_OK and the values that its plan gives alone.
"""
import threading

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


# two kinds in turn: blocks at the first basis vector only, and blocks over a long basis; low and high
# orders of the column passes (their shared memory exceeds 48 KB at N = 1024)
@pytest.mark.parametrize("N,L,rounds,kinds", [
    (256, 5.0, 600, (dict(restart=4), dict(restart=64))),
    (1024, 10.0, 15, (dict(restart=4, M=0), dict(restart=32, M=16))),
])
def test_direct_launches_from_several_threads(N, L, rounds, kinds):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    Q = wl.gaussian_mixture(N, L, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([2.5, 1.4 + 0.5j]))
    nt = 8
    plans = [dbar.Plan(N, L, prec="mixed", graphs=0, tol=1e-11, max_batch=1, autotune=0, sstep=4, inner_tol=1e-7,
                       max_outer=100, **kinds[i % 2]) for i in range(nt)]
    k = np.array([1.5 + 0.4j])
    alone = [p.solve(Q, k, want_m=False) for p in plans]
    assert all(a["status"] == dbar.DBAR_OK for a in alone)
    streams = [torch.cuda.Stream() for _ in plans]
    failed = []

    def work(i):
        try:
            for r in range(rounds):
                got = plans[i].solve(Q, k, want_m=False, stream=streams[i])
                if got["status"] != dbar.DBAR_OK or not np.array_equal(got["S"], alone[i]["S"]):
                    failed.append((i, r, got["status"]))
                    return
        except Exception as e:  # a refused launch raises in the thread
            failed.append((i, str(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(nt)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
