"""Work of another stream beside a long call of the persistent step: on grids
of more than 4 tiles per resident block every step is a launch of its own, so
a small solver's step waits for the step that runs, not for the whole call.

Bound: at most the running step and its own (shorter than one of the large
grid's), doubled for the two launches' scheduling: 4 large steps of the 24 in
flight. The large call's result is that of the same steps called one by one.
"""
import time

import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,mixed", [(1001, 503, False), (1001, 503, True), (1701, 1001, False)])
def test_a_small_step_does_not_wait_for_the_whole_call(nx, nz, mixed):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    steps = 24

    def solver(nx, nz, mixed=False):
        st = torch.cuda.Stream()
        grid = W.Grid(nx, nz, 20000.0, 10000.0)
        c = W.Constants(dt=0.05)
        s = G.Solver(grid, c, stream=st, mixed=mixed)
        s.set_conservative(W.random_flow(grid, c, seed=nx, uamp=2.0, thamp=1.0).fields)
        return s, st
    (big, _), (small, st) = solver(nx, nz, mixed), solver(160, 80)
    assert big.stats()["driver"].endswith("persistent") and small.stats()["driver"] == "persistent"
    big.step(2)
    small.step(2)
    waits = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        big.step_async(steps)
        small.step_async(1)
        st.synchronize()
        waits.append(time.perf_counter() - t0)
        torch.cuda.synchronize()
        one = (time.perf_counter() - t0) / steps
    big.sync()
    small.sync()
    print(nx, nz, mixed, "wait", min(waits), "step", one)
    assert min(waits) < 4 * one
    ref, _ = solver(nx, nz, mixed)
    for _ in range(2 + 3 * steps):
        ref.step(1)
    a, b = big.get_full(), ref.get_full()
    assert all(np.array_equal(a[k], b[k]) for k in a)
