"""Device arrays that end before the grid does, handed to the C interface: the
one-kernel paths of set_state and get_state leave them to the runtime's
copies, which refuse a range beyond its allocation. The arrays lie directly
before another allocation of this test, so that even an access past their end
would meet live memory; its bytes stay as they were."""
import ctypes as C

import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
BLOCK = 65536
NX, NZ = 64, 130   # 66,560 bytes a field: two rows more than a block holds


def test_short_device_arrays_are_refused():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    blocks = []
    for _ in range(16):
        p = C.c_uint64()
        assert cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(BLOCK)) == 0
        assert cu.cuMemsetD8_v2(p, 0xA5, C.c_size_t(BLOCK)) == 0
        blocks.append(p.value)
    pairs = [a for a in blocks if a + BLOCK in blocks]
    try:
        if not pairs:
            pytest.skip("no two adjacent allocations")
        short, guard = pairs[0], pairs[0] + BLOCK
        grid = W.Grid(NX, NZ, 40.0 * NX, 30.0 * NZ)
        wl = W.random_flow(grid, W.Constants(dt=0.2, mu=1.5), seed=7, uamp=3.0, thamp=2.0)
        dev = {k: torch.tensor(v, device="cuda") for k, v in wl.fields.items()}
        a, b = (G.Solver(grid, wl.const) for _ in range(2))
        a.set_conservative(dev)
        b.set_conservative(wl.fields)
        a.step(1)
        b.step(1)
        full = {k: torch.zeros(v.shape, dtype=torch.float64, device="cuda") for k, v in a.get_full().items()}
        a.get_full(full)

        def view(kind, arrays, **over):
            v = G._View()
            v.kind, v.mem = kind, G.MEM_DEVICE
            for k, t in arrays.items():
                setattr(v, k, t.data_ptr())
            for k, p in over.items():
                setattr(v, k, p)
            return C.byref(v)
        scratch = {k: torch.empty_like(t) for k, t in full.items()}
        for kind, arrays, name in ((G.STATE_FULL, scratch, "T"), (G.STATE_CONSERVATIVE, dev, "rhow")):
            keep = {k: t.clone() for k, t in arrays.items()}
            assert a.lib.gea_get_state(a.h, view(kind, keep, **{name: short})) == G.GEA_ERR_CUDA, name
        got = np.empty(BLOCK, dtype=np.uint8)
        assert cu.cuMemcpyDtoH_v2(C.c_void_p(got.ctypes.data), C.c_uint64(guard), C.c_size_t(BLOCK)) == 0
        assert (got == 0xA5).all()
        # the state is still there, and the next step is that of the other context
        a.step(1)
        b.step(1)
        x, y = a.get_full(), b.get_full()
        assert all(np.array_equal(x[k], y[k]) for k in x)
        for kind, arrays, name in ((G.STATE_FULL, full, "T"), (G.STATE_CONSERVATIVE, dev, "rhow")):
            assert a.lib.gea_set_state(a.h, view(kind, arrays, **{name: short})) == G.GEA_ERR_CUDA, name
        a.set_conservative(dev)
        b.set_conservative(wl.fields)
        a.step(1)
        b.step(1)
        x, y = a.get_full(), b.get_full()
        assert all(np.array_equal(x[k], y[k]) for k in x)
    finally:
        torch.cuda.synchronize()
        for p in blocks:
            cu.cuMemFree_v2(C.c_uint64(p))
