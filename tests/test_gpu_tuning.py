"""Tuned shapes belong to the kernels that were timed.

A server's lane gives every slot a potential of its own; the column variant that loads one potential's tables for
two slots does not exist there.  Lane and plan of one size keep their own timings.
"""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_lanes_and_plans_are_tuned_apart():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1508_02363_gb300 import dbar
    create = dbar._lib["_Z14plan_create_exPK11dbar_paramsibPP9dbar_plan"]  # how a server's lane makes its plan
    create.argtypes = [ctypes.POINTER(dbar.dbar_params), ctypes.c_int, ctypes.c_bool, ctypes.POINTER(ctypes.c_void_p)]
    p, lane = dbar.dbar_params_init(128, 5.0, prec="mixed", max_batch=13), ctypes.c_void_p()
    assert create(ctypes.byref(p), 1, True, ctypes.byref(lane)) == dbar.DBAR_OK
    variant, ms = dbar.dbar_plan_tuning(lane)
    plan = dbar.Plan(128, 5.0, prec="mixed", max_batch=13)
    _, own = dbar.dbar_plan_tuning(plan.handle)
    dbar.dbar_plan_destroy(lane)
    assert variant != 2 and ms[2] == 0 and ms[0] > 0 and ms[1] > 0  # no two-slot variant to time
    assert all(t > 0 for t in own) and list(own) != list(ms)
