"""dbar_host_copy: every byte, from any number of threads, and no waiting for helper threads.

On a host whose cores are busy a thread that was just started may not run for a scheduler tick; a
copy that started helpers and joined them took 7 to 8 times a memmove of the same 4 MB there
(median of 100, this test's set-up).  A copy must not take much longer than the caller alone.
"""
import ctypes
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

from paper_1508_02363_gb300 import dbar


@pytest.mark.parametrize("n", [0, 1, 4095, 2 << 20, (2 << 20) + 1, (4 << 20) - 3, 9 << 20])
def test_copies_every_byte(n):
    src = np.random.default_rng(n).integers(0, 256, n + 64, dtype=np.uint8)
    dst = np.zeros(n + 64, np.uint8)
    dbar.dbar_host_copy(dst.ctypes.data + 32, src.ctypes.data + 32, n)
    assert np.array_equal(dst[32:32 + n], src[32:32 + n]) and not dst[:32].any() and not dst[32 + n:].any()


def test_copies_from_several_threads():
    n, bad = 5 << 20, []

    def work(i):
        src, dst = np.full(n, i + 1, np.uint8), np.zeros(n, np.uint8)
        for _ in range(20):
            dst[:] = 0
            dbar.dbar_host_copy(dst.ctypes.data, src.ctypes.data, n)
            if not np.array_equal(dst, src):
                bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


def test_busy_cores_do_not_hold_up_a_copy():
    n = 4 << 20
    src, dst = np.ones(n, np.uint8), np.zeros(n, np.uint8)

    def median(f):
        t = []
        for _ in range(100):
            a = time.perf_counter()
            f()
            t.append(time.perf_counter() - a)
            time.sleep(0.0005)
        return sorted(t)[50]

    spin = [subprocess.Popen([sys.executable, "-c", "while True: pass"]) for _ in range(2 * os.cpu_count())]
    try:
        time.sleep(0.5)
        best = 1e9
        for _ in range(3):  # the quietest of three
            copy = median(lambda: dbar.dbar_host_copy(dst.ctypes.data, src.ctypes.data, n))
            best = min(best, copy / median(lambda: ctypes.memmove(dst.ctypes.data, src.ctypes.data, n)))
    finally:
        for p in spin:
            p.kill()
        for p in spin:
            p.wait()
    assert best < 3.0, best
