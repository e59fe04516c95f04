"""State in and out through device arrays (one kernel for all fields) against
the host copies, bit for bit: sizes with a last column or row of faces of
their own tile, both state slots (after an even and an odd number of steps),
K^{n-1} in the literal reading, a view with fields left out, and overlapping
destinations, which take the copies."""
import ctypes as C

import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    return torch, G


@pytest.mark.parametrize("nx,nz", [(4, 4), (32, 8), (33, 17), (63, 24)])
@pytest.mark.parametrize("lagged", [0, 1])
def test_device_arrays_equal_host_arrays(env, nx, nz, lagged):
    torch, G = env
    grid = W.Grid(nx, nz, 40.0 * nx, 30.0 * nz)
    wl = W.random_flow(grid, W.Constants(dt=0.2, mu=1.5, reading_flags=lagged), seed=nx + nz, uamp=3.0, thamp=2.0)
    dev = {k: torch.tensor(v, device="cuda") for k, v in wl.fields.items()}
    a, b = (G.Solver(grid, wl.const) for _ in range(2))
    a.set_conservative(wl.fields)
    b.set_conservative(dev)
    for steps in (0, 1, 1):
        a.step(steps)
        b.step(steps)
        host = a.get_full()
        out = {k: torch.full(v.shape, float("nan"), dtype=torch.float64, device="cuda") for k, v in host.items()}
        b.get_full(out)
        cons = {k: torch.full((nz, nx), float("nan"), dtype=torch.float64, device="cuda") for k in wl.fields}
        b.get_conservative(cons)
        chost = a.get_conservative()
        for k in host:
            assert np.array_equal(out[k].cpu().numpy(), host[k]), (k, steps)
        for k in chost:
            assert np.array_equal(cons[k].cpu().numpy(), chost[k]), (k, steps)
        # a full set from device arrays continues as one from host arrays
        a.set_full(host)
        b.set_full(out)
    # fields left out, and a destination given twice
    v = G._View()
    v.kind, v.mem = G.STATE_FULL, G.MEM_DEVICE
    one = torch.full((nz, nx), float("nan"), dtype=torch.float64, device="cuda")
    v.T = one.data_ptr()
    assert b.lib.gea_get_state(b.h, C.byref(v)) == G.GEA_OK
    assert np.array_equal(one.cpu().numpy(), a.get_full()["T"])
    v.h = one.data_ptr()
    assert b.lib.gea_get_state(b.h, C.byref(v)) == G.GEA_OK
    assert np.array_equal(one.cpu().numpy(), a.get_full()["h"])
