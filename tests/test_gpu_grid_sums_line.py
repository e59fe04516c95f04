"""Grid reductions of the persistent step at the number of blocks where they
change form: up to 64 blocks one warp adds a value's partial sums straight
from memory, above that all threads do. One tile of 32 x 8 cells is one block
here; the oracle adds in another order: the repository's bar of 1e-10 relative
L2, velocities against the norm of their vector. Mixed precision: the bars of
its other tests (scalars 5e-9, velocities 5e-7)."""
import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# blocks: 63, 64, 65, 96
@pytest.mark.parametrize("nx,nz", [(63 * 32, 8), (256, 64), (65 * 32, 7), (380, 60)])
@pytest.mark.parametrize("mixed", [False, True], ids=["fp64", "mixed"])
def test_against_oracle(oracle_mod, nx, nz, mixed):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    grid = W.Grid(nx, nz, 35.0 * nx, 30.0 * nz)
    c = W.Constants(dt=0.2, n_corr=2, mu=1.5)
    wl = W.random_flow(grid, c, seed=nx * 1000 + nz, uamp=3.0, thamp=2.0)
    o = oracle_mod.Oracle(grid, c)
    so = o.derive(wl.fields)
    o.step(so, 3)
    s = G.Solver(grid, c, mixed=mixed)
    s.set_conservative(wl.fields)
    s.step(3)
    st = s.stats()
    assert st["status"] == 0 and st["driver"].endswith("persistent"), st
    g = s.get_full()
    for k in ("rho", "T", "h", "p", "pp"):
        assert np.linalg.norm(g[k] - so[k]) <= (5e-9 if mixed else 1e-10) * np.linalg.norm(so[k]), k
    size = np.hypot(np.linalg.norm(so["u"]), np.linalg.norm(so["w"]))
    for k in ("u", "w"):
        assert np.linalg.norm(g[k] - so[k]) <= (5e-7 if mixed else 1e-10) * size, k
