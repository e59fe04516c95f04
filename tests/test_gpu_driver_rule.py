"""The choice of the step driver at its line (16 tiles of 32 x 8 cells per
resident block, 8 in mixed precision): the largest grid of the persistent step
and the next row of tiles, and an odd grid between. The two drivers run the
same phases: they agree to the order of the reduction sums (FP64 1e-11 of the
field, mixed 1e-8, the bars of the tile-column tests)."""
import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,mixed,persistent", [
    (3072, 608, False, True), (3072, 616, False, False), (1001, 503, False, True),
    (3072, 304, True, True), (3072, 312, True, False), (1001, 503, True, True)])
def test_drivers_agree_at_the_line(nx, nz, mixed, persistent):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line is that of 152 SMs")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    grid = W.Grid(nx, nz, 30.0 * nx, 12000.0)
    c = W.Constants(dt=0.05, mu=1.5)
    wl = W.random_flow(grid, c, seed=nx + nz, uamp=3.0, thamp=2.0)
    out = []
    for graph in (False, True):
        s = G.Solver(grid, c, graph=graph, mixed=mixed)
        s.set_conservative(wl.fields)
        s.step(2)
        st = s.stats()
        want = ("mixed_" if mixed else "") + "persistent" if persistent and not graph else ("mixed" if mixed else "graph")
        assert st["status"] == 0 and st["driver"] == want, st
        out.append(s.get_full())
        s.close()
    a, b = out
    vel = np.hypot(np.linalg.norm(b["u"]), np.linalg.norm(b["w"]))
    for k in ("rho", "T", "pp", "u", "w"):
        scale = vel if k in "uw" else np.linalg.norm(b[k])
        assert np.linalg.norm(a[k] - b[k]) <= (1e-8 if mixed else 1e-11) * scale, k
