"""The kernels' reciprocal (Chebyshev's third-order iteration from the
hardware seed) against correctly rounded divisions, through the fields it
forms: the Helmholtz reaction term c = 1 / (R T dt) and the face coefficients
D_f = dt (rho2_a + rho2_b) / (rho1_a + rho1_b).

Bounds, in units of 2^-53 of the value: the reciprocal is within 2 (one ulp),
R T and the factor 1 / dt (itself rounded) add 1 each: 5 for c. For D: the two
factors dt rho2 and their sum 2, the sum of the rho1 1, the reciprocal 2, the
product 1, and the reference's own roundings 3: 9."""
import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("nx,nz,dt", [(4, 4, 0.2), (65, 33, 0.3), (160, 80, 0.1)])
@pytest.mark.parametrize("graph", [False, True], ids=["persistent", "graph"])
def test_reciprocal_is_within_an_ulp(nx, nz, dt, graph):
    import torch
    assert torch.cuda.is_available(), "CUDA device required"
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    grid = W.Grid(nx, nz, 120.0 * nx, 120.0 * nz)
    wl = W.random_flow(grid, W.Constants(dt=dt, mu=1.5), seed=nx + nz, uamp=3.0, thamp=20.0)
    s = G.Solver(grid, wl.const, graph=graph)
    s.set_conservative(wl.fields)
    s.step(2)
    T, r1, r2 = s.get_full()["T"], s.field("rho1"), s.field("rho2")
    c = 1.0 / (wl.const.R * T) / dt
    assert np.abs(s.field("hc") / c - 1.0).max() <= 5 * U + 2 * U   # the quotient's own rounding
    for name, ax in (("Dx", 1), ("Dz", 0)):
        D = s.field(name)
        inner = D[:, 1:-1] if ax else D[1:-1]
        a, b = (np.take(r2, range(0, r2.shape[ax] - 1), ax), np.take(r2, range(1, r2.shape[ax]), ax))
        p, q = (np.take(r1, range(0, r1.shape[ax] - 1), ax), np.take(r1, range(1, r1.shape[ax]), ax))
        assert np.abs(inner / (dt * (a + b) / (p + q)) - 1.0).max() <= 9 * U + 2 * U, name
