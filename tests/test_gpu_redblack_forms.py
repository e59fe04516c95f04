"""Forms of the red-black pressure solve beside those of
tests/test_gpu_redblack.py, against the oracle: damped and over-relaxed black
cells in mixed precision, and a network attached (initial guess,
preconditioner, both) with one to four correctors, whose solves start from
buffers that alternate.

The converged pressure depends on neither, so the repository's bars hold: FP64
1e-10 relative L2 (velocities against the norm of their vector); mixed
precision 5e-9 for the scalars and 5e-7 for the velocities, with two and more
correctors as everywhere.
"""
import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gea():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    return G


def compare(oracle_mod, s, wl, steps, mixed):
    o = oracle_mod.Oracle(wl.grid, wl.const)
    so = o.derive(wl.fields)
    o.step(so, steps)
    s.set_conservative(wl.fields)
    s.step(steps)
    assert s.stats()["status"] == 0
    g = s.get_full()
    for k in ("rho", "T", "h", "p", "pp"):
        assert np.linalg.norm(g[k] - so[k]) <= (5e-9 if mixed else 1e-10) * np.linalg.norm(so[k]), k
    size = np.hypot(np.linalg.norm(so["u"]), np.linalg.norm(so["w"]))
    for k in ("u", "w"):
        assert np.linalg.norm(g[k] - so[k]) <= (5e-7 if mixed else 1e-10) * size, k


@pytest.mark.parametrize("graph", [False, True], ids=["persistent", "graph"])
@pytest.mark.parametrize("nx,nz,mgmin,ncorr,omega", [(132, 20, 200, 3, 0.8), (72, 40, 50, 2, 1.15), (65, 7, 0, 2, 1.2),
                                                     (128, 16, 64, 2, 1.6)])
def test_mixed_with_a_smoother_weight(gea, oracle_mod, nx, nz, mgmin, ncorr, omega, graph):
    grid = W.Grid(nx, nz, 35.0 * nx, 30.0 * nz)
    c = W.Constants(dt=0.2, n_corr=ncorr, mu=1.5)
    wl = W.random_flow(grid, c, seed=nx * 1000 + nz, uamp=3.0, thamp=2.0)
    s = gea.Solver(grid, c, mg_min_cells=mgmin, graph=graph, mixed=True)
    s.set_smoother_weight(omega)
    compare(oracle_mod, s, wl, 5, True)


@pytest.mark.parametrize("mode,mixed,ncorr", [(m, False, n) for m in (1, 2, 3) for n in (1, 3, 4)] +
                         [(1, True, 3), (1, True, 4)])
@pytest.mark.parametrize("mgmin", [0, 200], ids=["default", "levels"])
def test_network_with_correctors(gea, oracle_mod, mode, mixed, ncorr, mgmin):
    from paper_2303_10499_gb300 import learned
    grid = W.Grid(128, 64, 35.0 * 128, 30.0 * 64)
    c = W.Constants(dt=0.2, n_corr=ncorr, mu=1.5)
    wl = W.random_flow(grid, c, seed=128064, uamp=3.0, thamp=2.0)
    net = gea.Net(1, 64, 128, relu=False)
    net.set_params(learned.initial_params(3))
    s = gea.Solver(grid, c, mg_min_cells=mgmin, mixed=mixed)
    s.attach_net(net, mode)
    compare(oracle_mod, s, wl, 4, mixed)
