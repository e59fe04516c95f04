"""The preconditioner that the pressure solve's CG runs on: the black half of one
V(1,1)-cycle with a red-black Gauss-Seidel smoother.

CG needs it linear, symmetric and positive definite; an asymmetric one would
only slow CG down, which a parity test does not see. Three checks:

* gea_apply_precond (the cycle on all cells) is linear, symmetric and positive
  for every weight of the black relaxations (1e-12, the bound of
  tests/test_gpu_multigrid.py).
* For a residual that is zero on the red cells its black part is what CG's own
  kernels (the start of a solve and the iterations, which work on the black
  half) made of the same residual: the residual and z = M r of the last
  iteration are read from the context's arrays (debug_pads tells where they
  are). Both sides form the same sums in another order: 1e-12 of the largest
  value. The black half of a symmetric positive operator is symmetric and
  positive.
* CG's iteration counts on fixed multi-level problems, in both precisions, in
  two and three dimensions, are at most one above those of the present cycle.
"""
import ctypes as C

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


def workload(nx, nz, **kw):
    grid = W.Grid(nx, nz, 35.0 * nx, 30.0 * nz)
    return W.random_flow(grid, W.Constants(dt=0.2, mu=1.5, **kw), seed=nx * 1000 + nz, uamp=3.0, thamp=2.0)


def array(s, name):
    """A context array (rows x pitch) as it lies in device memory."""
    r = next(x for x in s.debug_pad_regions() if x["name"] == name)
    out = np.empty((r["rows"], r["pitch"]))
    assert C.CDLL("libcuda.so.1").cuMemcpyDtoH_v2(C.c_void_p(out.ctypes.data), C.c_uint64(r["ptr"]),
                                                  C.c_size_t(out.nbytes)) == 0
    return out


# nx, nz, mg_min_cells, levels
GRIDS = [(132, 20, 200, 3), (72, 40, 50, 4), (96, 64, 3000, 2), (160, 80, 200, 4)]


@pytest.mark.parametrize("omega", [1.0, 0.8, 1.15, 1.6])
@pytest.mark.parametrize("nx,nz,mgmin,levels", GRIDS)
def test_cycle_linear_symmetric_positive(gea, nx, nz, mgmin, levels, omega):
    wl = workload(nx, nz)
    s = gea.Solver(wl.grid, wl.const, mg_min_cells=mgmin)
    s.set_conservative(wl.fields)
    s.set_smoother_weight(omega)
    s.step(2)
    assert s.stats()["mg_levels"] == levels
    rng = np.random.default_rng(nx + nz)
    for smooth in (False, True):
        x, y = rng.standard_normal((2, nz, nx))
        if smooth:   # smooth vectors reach the coarse levels
            x, y = (np.cumsum(np.cumsum(v, 0), 1) for v in (x, y))
        mx, my = s.apply_precond(x), s.apply_precond(y)
        sym = abs(np.vdot(x, my) - np.vdot(y, mx))
        assert sym <= 1e-12 * np.linalg.norm(x) * np.linalg.norm(my), (smooth, sym)
        assert np.vdot(x, mx) > 0 and np.vdot(y, my) > 0
        lin = s.apply_precond(x + 2.0 * y) - (mx + 2.0 * my)
        assert np.abs(lin).max() <= 1e-12 * (np.abs(mx).max() + 2.0 * np.abs(my).max()), smooth


@pytest.mark.parametrize("graph", [False, True], ids=["persistent", "graph"])
@pytest.mark.parametrize("omega", [1.0, 0.8, 1.15, 1.6])
@pytest.mark.parametrize("nx,nz,mgmin,levels", GRIDS + [(65, 33, 0, 1), (160, 80, 10 ** 6, 1)])
@pytest.mark.parametrize("iterations", ["start", "several"])
def test_black_half_is_that_of_the_cycle(gea, nx, nz, mgmin, levels, omega, graph, iterations):
    def solved(rtol):
        wl = workload(nx, nz, n_corr=1, cg_rtol=rtol)
        s = gea.Solver(wl.grid, wl.const, mg_min_cells=mgmin, graph=graph, debug_pads=True)
        s.set_conservative(wl.fields)
        s.set_smoother_weight(omega)
        s.step(1)
        return s, s.stats()
    # "start": a tolerance just below the residual that the solve starts from
    # (reported by a solve with nothing to do), so that one iteration is enough
    # and z comes from the start
    s, st = solved(1e-17 if iterations == "several" else 0.99 * solved(0.5)[1]["cg_relres"][0])
    n = st["cg_iters"][0]
    assert st["status"] == 0 and st["mg_levels"] == levels and (n >= 3 if iterations == "several" else n == 1), st
    # a multi-level solve ends before the cycle on its last residual; one level
    # updates z with the residual, in place
    rb = array(s, "L0.e" if levels == 1 or (n - 1) % 2 == 0 else "L0.r_alt")
    z = array(s, "L0.e2")
    full, black = np.zeros((nz, nx)), []
    for k in range(nz):
        cols = np.arange(k & 1, nx, 2)
        full[k, cols] = rb[k, :cols.size]
        black.append(z[k, :cols.size])
    got = s.apply_precond(full)
    scale = max(np.abs(b).max() for b in black)
    assert scale > 0
    for k in range(nz):
        d = np.abs(got[k, (k & 1)::2] - black[k]).max()
        assert d <= 1e-12 * scale, (k, d / scale)


@pytest.mark.parametrize("mixed,most", [(False, (16, 11)), (True, (7, 7))], ids=["fp64", "mixed"])
def test_iterations_2d(gea, mixed, most):
    """Five levels at 2.5 m."""
    grid, c = W.Grid(400, 400, 1000.0, 1000.0), W.Constants(dt=0.1)
    s = gea.Solver(grid, c, mixed=mixed)
    s.set_conservative(W.random_flow(grid, c, seed=1, uamp=2.0, thamp=1.0).fields)
    s.step(3)
    st = s.stats()
    assert st["mg_levels"] == 5 and all(a <= b for a, b in zip(st["cg_iters"], most)), st


@pytest.mark.parametrize("n,dt,mgmin,levels,mixed,most", [
    ((96, 96, 96), 0.5, 0, 5, False, (24, 20)), ((96, 96, 96), 0.5, 0, 5, True, (10, 11)),
    ((96, 64, 64), 0.2, 100, 5, False, (21, 17)), ((96, 64, 64), 0.2, 100, 5, True, (9, 9))])
def test_iterations_3d(gea, n, dt, mgmin, levels, mixed, most):
    grid, c = W.Grid3(*n, *(20.0 * m for m in n)), W.Constants(dt=dt)
    s = gea.Solver3D(grid, c, mg_min_cells=mgmin, mixed=mixed)
    s.set_conservative(W.random_flow3(grid, c, seed=1, uamp=2.0, thamp=1.0).fields)
    s.step(2)
    st = s.stats()
    assert st["mg_levels"] == levels and all(a <= b for a, b in zip(st["cg_iters"], most)), st
