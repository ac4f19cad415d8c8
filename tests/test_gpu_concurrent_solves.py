"""Solves of several contexts on several threads of one process.

The resident iteration of small lattices holds most of the SMs for milliseconds
at a time; while calls of other threads need the device, a solve runs the four
kernels of an iteration, which share it.  Both give the same bits, so what is
checked is the solutions against solo ones and, by the number of kernels
launched, which form ran."""
import threading
import time

import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


def _context(gpu, dims, seed):
    c = gpu.Context(dims)
    c.links_upload(inputs.random_links(dims, seed=seed))
    return c, inputs.gaussian_field(dims, k=seed)


def _resident(info):
    return info["kernel_launches"] < info["iters"]   # four launches per iteration otherwise


def test_small_solve_shares_the_device_with_another_threads_call(gpu):
    c, b = _context(gpu, (12, 12, 12, 12), 1)
    big, bb = _context(gpu, (24, 24, 24, 24), 2)
    sh = inputs.log_shifts(3)
    x0, i0 = c.mscg_solve(0.05, sh, 1e-10, b)
    assert _resident(i0), "alone on the device the resident iteration runs"
    stop, started, err = threading.Event(), threading.Event(), []

    def busy():
        try:
            while not stop.is_set():
                started.set()
                big.mscg_solve(0.01, sh, 1e-10, bb)
        except Exception as e:
            err.append(e)
            started.set()

    t = threading.Thread(target=busy)
    t.start()
    started.wait()
    time.sleep(0.05)   # inside the first of the long solves (0.1 s and more)
    try:
        x1, i1 = c.mscg_solve(0.05, sh, 1e-10, b)
    finally:
        stop.set()
        t.join()
    assert not err
    assert np.array_equal(x0, x1) and i0["iters"] == i1["iters"] and i0["true_resid"] == i1["true_resid"]
    assert not _resident(i1), "the resident iteration ran beside another thread's solve"
    time.sleep(0.2)
    x2, i2 = c.mscg_solve(0.05, sh, 1e-10, b)
    assert _resident(i2) and np.array_equal(x0, x2)
    c.close()
    big.close()


@pytest.mark.parametrize("dims,n", [((8, 8, 8, 8), 2), ((8, 8, 8, 8), 6), ((12, 12, 12, 12), 3), ((16, 16, 16, 16), 2)])
def test_solves_on_threads_equal_solo(gpu, dims, n):
    """Batches that fit beside one another (two of 64 SMs) and that do not."""
    ctxs = [_context(gpu, dims, 10 + k) for k in range(n)]
    sh = inputs.log_shifts(3)
    solo = [c.mscg_solve(0.05, sh, 1e-10, b) for c, b in ctxs]
    got, err = [[] for _ in range(n)], []

    def work(k):
        try:
            for _ in range(3):
                got[k].append(ctxs[k][0].mscg_solve(0.05, sh, 1e-10, ctxs[k][1]))
        except Exception as e:
            err.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(n)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not err
    for k in range(n):
        for x, info in got[k]:
            assert np.array_equal(x, solo[k][0]) and info["true_resid"] == solo[k][1]["true_resid"]
    for c, _ in ctxs:
        c.close()
