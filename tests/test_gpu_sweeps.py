"""The basis sweeps' shared-memory stages: bulk copies refill a stage that the threads have read.

A barrier does not order a read through the generic proxy before a bulk copy's write (async
proxy): every kernel that refills a stage has its readers pass a proxy fence first (checked in the
source, on the CPU).  On the GPU: sweeps over more basis vectors than there are stages give the
same values in every run, with one and four elements per thread, in FP32 and FP64.
"""
import os
import re

import numpy as np
import pytest

import workloads as wl

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_02363_gb300", "csrc")


def test_refilled_stages_are_released_by_a_proxy_fence():
    text = open(os.path.join(CSRC, "krylov.cuh")).read()
    kernels = [k for k in re.split(r"(?=^(?:template <[^\n]*>\n)?(?:static )?__global__ )", text, flags=re.M) if "bulk_g2s(stage" in k]
    assert len(kernels) == 2
    for k in kernels:
        # between the stage's last read and the barrier before its refill
        assert re.search(r"stage_release\(\);\s*__syncthreads\(\);[^;]*?\n\s*if \(threadIdx\.x == 0", k), k[:200]


@pytest.mark.gpu
@pytest.mark.parametrize("N,prec,restart", [(64, "mixed", 32), (64, "fp64", 32), (256, "mixed", 32), (256, "fp64", 16)])
def test_sweeps_repeat_value_for_value(N, prec, restart):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    Q = wl.gaussian_mixture(N, 5.0, np.array([[0.3, -0.2], [-0.9, 0.6]]), np.array([1.1, 0.9]), np.array([2.5, 1.4 + 0.5j]))
    k = 1.5 * np.exp(0.4j * np.arange(16))
    plan = dbar.Plan(N, 5.0, prec=prec, restart=restart, inner_tol=1e-7, tol=1e-12, max_batch=16)
    ref = plan.solve(Q, k, want_m=False)
    assert ref["status"] == dbar.DBAR_OK and np.all(ref["iters"][:, 0] > 8)
    for _ in range(8):
        r = plan.solve(Q, k, want_m=False)
        assert np.array_equal(r["S"], ref["S"]) and np.array_equal(r["iters"], ref["iters"])
