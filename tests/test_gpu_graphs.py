"""Captured cycles are kept for every way in which a program uses a plan."""
import time

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,prec", [(128, "mixed")])
def test_alternating_guesses_do_not_capture_again(N, prec):
    # plain solves and solves from a guess in turn take the time of each kind on its own (1.27 times that when
    # every call captured its cycles again)
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    Q = torch.from_numpy(wl.gaussian_mixture(N, 5.0, np.array([[0.3, -0.2]]), np.array([1.1]), np.array([1.4]))).cuda()
    k = np.array([0.4 - 0.3j])
    S = torch.empty((1, N, N), dtype=torch.complex128, device="cuda")
    plan = dbar.Plan(N, 5.0, prec=prec, restart=32, tol=1e-12, max_batch=1)
    plan.solve_device(Q, k, S)
    x0 = 1.01 * S

    def plain():
        plan.solve_device(Q, k, S)

    def guess():
        plan.solve_device(Q, k, S, x0=x0)

    def seconds(f, g):
        best = 1e9
        for _ in range(5):
            a = time.perf_counter()
            for _ in range(10):
                f()
                g()
            best = min(best, time.perf_counter() - a)
        return best

    for f in (plain, guess):
        f(), f()
    alone = 0.5 * (seconds(plain, plain) + seconds(guess, guess))
    ratio = seconds(plain, guess) / alone
    print(f"N {N} {prec}: alone {alone / 20 * 1e3:.2f} ms a solve, in turn {ratio:.2f} times that")
    assert ratio < 1.12, ratio
