"""The work this library is measured on: time steps of the dry compressible
Euler solver through its public classes, and one training pass of the learned
pressure network.

A step case loads a state (set_conservative, device buffers), advances it and
reads the new state back (device buffers), as a program does that couples the
solver to something else on the GPU or restarts it from a field. States are
rising thermal bubbles in a neutral hydrostatic atmosphere that already move:
a smooth, mass-flux divergence-free flow of a few m/s is added, so that every
term of the step is active.
"""
import math

import numpy as np
import torch

from paper_2303_10499_gb300 import gea, learned
from paper_2303_10499_gb300.workloads import Constants, Grid, Grid3

DEVICE = "cuda"
THETA0 = 300.0


def listed():
    return [
        # a small run at its per-call cost: one step of the coarse 20 km bubble
        dict(name="bubble_160x80", kind="step2d", nx=160, nz=80, box="20km", dt=0.1, steps=1, mixed=False, cs=0.0),
        # the headline configuration, in double and in mixed precision
        dict(name="bubble_640x320", kind="step2d", nx=640, nz=320, box="20km", dt=0.05, steps=4, mixed=False, cs=0.0),
        dict(name="bubble_640x320_mixed", kind="step2d", nx=640, nz=320, box="20km", dt=0.05, steps=4, mixed=True,
             cs=0.0),
        # the paper's own 5 m grid
        dict(name="paper_200x200", kind="step2d", nx=200, nz=200, box="1km", dt=0.1, steps=4, mixed=False, cs=0.0),
        # odd sizes in both directions, between the small and the large grids
        dict(name="ragged_1001x503", kind="step2d", nx=1001, nz=503, box="20km", dt=0.05, steps=2, mixed=False,
             cs=0.0),
        # fields larger than the caches, in double and in mixed precision
        dict(name="bubble_4096x2048", kind="step2d", nx=4096, nz=2048, box="20km", dt=0.05, steps=1, mixed=False,
             cs=0.0),
        dict(name="bubble_4096x2048_mixed", kind="step2d", nx=4096, nz=2048, box="20km", dt=0.05, steps=1, mixed=True,
             cs=0.0),
        # one large-eddy simulation at 2.5 m
        dict(name="les_400x400", kind="step2d", nx=400, nz=400, box="1km", dt=0.1, steps=2, mixed=False, cs=0.17),
        # a batch of large-eddy simulations of three sizes in one launch
        dict(name="les_ensemble_24", kind="ensemble", members=24, n0=100, n1=200, n2=400, dt=0.1, steps=1,
             mixed=False, cs=0.17),
        # three dimensions: a medium run in mixed precision, the largest in double
        dict(name="bubble3d_192x192x96_mixed", kind="step3d", nx=192, ny=192, nz=96, dt=0.05, steps=1, mixed=True,
             cs=0.17),
        dict(name="bubble3d_512x512x256", kind="step3d", nx=512, ny=512, nz=256, dt=0.05, steps=1, mixed=False,
             cs=0.17),
        # one training pass of the pressure network at its default batch
        dict(name="network_8x256x256", kind="network", n=8, h=256, w=256),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step2d", "step2d", "step2d", "les", "ensemble", "step3d", "network"])
    if kind == "step2d":
        nx = _log_size(rng, 64, 4096)
        nz = max(32, min(2048, int(nx * rng.choice([0.5, 0.5, rng.uniform(0.35, 0.65)]))))
        if rng.random() < 0.6:   # most grids are chosen even, some are not
            nx, nz = nx // 8 * 8, max(32, nz // 8 * 8)
        return dict(kind="step2d", nx=nx, nz=nz, box="20km", dt=0.1 if nx < 400 else 0.05, steps=rng.randint(1, 4),
                    mixed=rng.random() < 0.35, cs=0.0)
    if kind == "les":
        n = _log_size(rng, 64, 512)
        if rng.random() < 0.7:
            n = n // 4 * 4
        return dict(kind="step2d", nx=n, nz=n, box="1km", dt=0.1, steps=rng.randint(1, 4), mixed=rng.random() < 0.35,
                    cs=rng.choice([0.0, 0.17]))
    if kind == "ensemble":
        return dict(kind="ensemble", members=rng.randint(3, 36), n0=rng.choice([50, 64, 100]),
                    n1=rng.choice([128, 150, 200]), n2=rng.choice([256, 320, 400]), dt=0.1, steps=1,
                    mixed=rng.random() < 0.35, cs=0.17)
    if kind == "step3d":
        nx, ny, nz = _log_size(rng, 33, 256), _log_size(rng, 33, 256), _log_size(rng, 24, 128)
        if rng.random() < 0.6:
            nx, ny, nz = nx // 4 * 4, ny // 4 * 4, nz // 4 * 4
        return dict(kind="step3d", nx=nx, ny=ny, nz=nz, dt=0.05, steps=1, mixed=rng.random() < 0.4,
                    cs=rng.choice([0.0, 0.17]))
    return dict(kind="network", n=rng.randint(1, 12), h=8 * rng.randint(8, 32), w=8 * rng.randint(8, 32))


# ---- inputs ----

def _constants(case):
    if case.get("box") == "1km" or case["kind"] == "ensemble":   # Section 4 of the paper: cv = 715.5, mu = 0.15 or 0.3
        return Constants(cp=287.0 + 715.5, dt=case["dt"], mu=0.3 if case["cs"] else 0.15, cs=case["cs"])
    return Constants(dt=case["dt"], cs=case["cs"])


def _background(nz, dz, c):
    """Neutral column in discrete hydrostatic balance: temperature and pressure at cell centres."""
    z = (np.arange(nz) + 0.5) * dz
    T = THETA0 - c.g * z / c.cp
    rho = np.empty(nz)
    rho[0] = c.p0 * (1.0 - c.g * z[0] / (c.cp * THETA0)) ** (c.cp / c.R) / (c.R * T[0])
    for k in range(nz - 1):
        rho[k + 1] = rho[k] * (c.R * T[k] - 0.5 * c.g * dz) / (c.R * T[k + 1] + 0.5 * c.g * dz)
    return T, rho * c.R * T


def _axis(n, length, dim, ndim):
    x = (torch.arange(n, dtype=torch.float64, device=DEVICE) + 0.5) * (length / n)
    return x.reshape([-1 if d == dim else 1 for d in range(ndim)])


def _bubble(sizes, lengths, c, amp, radius, centre, smooth, rng, speed):
    """Conservative fields of a bubble in the balanced background with a smooth flow whose mass flux has no
    divergence. sizes and lengths run over x, (y,) z; arrays over z, (y,) x."""
    nd = len(sizes)
    z = _axis(sizes[-1], lengths[-1], 0, nd)
    hor = [_axis(sizes[d], lengths[d], nd - 1 - d, nd) for d in range(nd - 1)]
    Tb, pb = _background(sizes[-1], lengths[-1] / sizes[-1], c)
    shape = [-1] + [1] * (nd - 1)
    Tb = torch.tensor(Tb, device=DEVICE).reshape(shape)
    pb = torch.tensor(pb, device=DEVICE).reshape(shape)
    r = torch.sqrt(sum((x - x0) ** 2 for x, x0 in zip(hor + [z], centre)))
    th = torch.where(r <= radius, 0.5 * amp * (1.0 + torch.cos(math.pi * r / radius)) if smooth else amp, 0.0)
    T = Tb * (THETA0 + th) / THETA0
    del r, th
    rho = pb / (c.R * T)
    flux = [torch.zeros_like(rho) for _ in range(nd)]
    for _ in range(3):
        wave = [float(rng.integers(1, 4)) * math.pi / length for length in lengths]
        for d in range(nd - 1):   # a stream function in the plane of direction d and z
            a = speed * rng.uniform(-1.0, 1.0)
            sin, cos, other = torch.sin(wave[d] * hor[d]), torch.cos(wave[d] * hor[d]), 1.0
            for e in range(nd - 1):
                if e != d:
                    other = other * torch.cos(wave[e] * hor[e])
            flux[d] -= a * sin * other * torch.cos(wave[-1] * z)
            flux[-1] += a * (wave[d] / wave[-1]) * cos * other * torch.sin(wave[-1] * z)
    kin = sum(f * f for f in flux) * 0.5 / rho
    names = ("rhou", "rhow") if nd == 2 else ("rhou", "rhov", "rhow")
    out = {"rho": rho, "rhoe": rho * (c.cv * T + c.g * z) + kin}
    out.update(zip(names, flux))
    return {k: v.contiguous() for k, v in out.items()}


def _step2d_inputs(case, nx, nz, seed):
    rng = np.random.default_rng(seed)
    c = _constants(case)
    if case.get("box", "1km") == "20km":
        grid = Grid(nx, nz, 20000.0, 10000.0)
        amp, radius, centre, smooth, speed = 2.0 * rng.uniform(0.8, 1.2), 2000.0, (10000.0, 2000.0), True, 2.0
    else:
        grid = Grid(nx, nz, 1000.0, 1000.0)
        amp, radius, centre, smooth, speed = rng.uniform(0.3, 0.7), 250.0, (500.0, 260.0), case["cs"] == 0.0, 1.0
    centre = tuple(x + 0.2 * radius * rng.uniform(-1.0, 1.0) for x in centre)
    return grid, c, _bubble((nx, nz), (grid.lx, grid.lz), c, amp, radius, centre, smooth, rng, speed)


def _step3d_inputs(case, seed):
    rng = np.random.default_rng(seed)
    c = _constants(case)
    grid = Grid3(case["nx"], case["ny"], case["nz"], 10000.0, 10000.0, 10000.0)
    centre = tuple(x + 400.0 * rng.uniform(-1.0, 1.0) for x in (5000.0, 5000.0, 2000.0))
    f = _bubble((grid.nx, grid.ny, grid.nz), (grid.lx, grid.ly, grid.lz), c, 2.0 * rng.uniform(0.8, 1.2), 2000.0,
                centre, True, rng, 2.0)
    return grid, c, f


def _member_sizes(case):
    return [case["n%d" % (m % 3)] for m in range(case["members"])]


def _network_inputs(case, seed):
    """Residual and Helmholtz operator batches: smooth residuals with some noise, coefficients near those of the
    fine bubbles, closed at the walls."""
    n, h, w = case["n"], case["h"], case["w"]
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)

    def rnd(*shape):
        return torch.randn(shape, generator=g, device=DEVICE)
    y, x = torch.arange(h, device=DEVICE)[:, None] / h, torch.arange(w, device=DEVICE)[None, :] / w
    r = 0.05 * rnd(n, h, w)
    for m in range(1, 5):
        r += rnd(n, 1, 1) * torch.cos(m * math.pi * x) * torch.cos((5 - m) * math.pi * y) / m
    c = 1.0 + 0.05 * torch.cos(math.pi * y) + 0.01 * rnd(n, h, w)
    ax, az = 9.0 + 0.1 * rnd(n, h, w + 1), 9.0 + 0.1 * rnd(n, h + 1, w)
    ax[:, :, 0] = ax[:, :, -1] = 0.0
    az[:, 0] = az[:, -1] = 0.0
    theta = learned.initial_params(seed)
    return r, c.contiguous(), ax, az, theta


def _empty(shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device=DEVICE)


def _full_out(grid):
    out = {k: _empty((grid.nz, grid.nx)) for k in gea.FULL_FIELDS[:-1]}
    out["phix"], out["phiz"] = _empty((grid.nz, grid.nx + 1)), _empty((grid.nz + 1, grid.nx))
    return out


def _ensemble_out(grids):
    """Each member's fields as views into one buffer per field."""
    flat, outs = {}, [{} for _ in grids]
    for k in gea.FULL_FIELDS[:-1]:
        shapes = [(g.nz, g.nx + 1) if k == "phix" else (g.nz + 1, g.nx) if k == "phiz" else (g.nz, g.nx) for g in grids]
        flat[k] = _empty(sum(a * b for a, b in shapes))
        at = 0
        for o, (a, b) in zip(outs, shapes):
            o[k] = flat[k][at:at + a * b].view(a, b)
            at += a * b
    return outs, flat


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    if case["kind"] == "step2d":
        grid, c, f = _step2d_inputs(case, case["nx"], case["nz"], seed)
        s = gea.Solver(grid, c, stream=stream, mixed=case["mixed"])
        return {"kind": "step", "solver": s, "fields": f, "out": _full_out(grid), "steps": case["steps"]}
    if case["kind"] == "step3d":
        grid, c, f = _step3d_inputs(case, seed)
        s = gea.Solver3D(grid, c, stream=stream, mixed=case["mixed"])
        out = {k: _empty((grid.nz, grid.ny, grid.nx)) for k in gea.STATE3_FIELDS}
        return {"kind": "step", "solver": s, "fields": f, "out": out, "steps": case["steps"]}
    if case["kind"] == "ensemble":
        solvers, fields = [], []
        for m, n in enumerate(_member_sizes(case)):
            grid, c, f = _step2d_inputs(case, n, n, 1000 * seed + m)
            solvers.append(gea.Solver(grid, c, stream=stream, mixed=case["mixed"]))
            fields.append(f)
        outs, flat = _ensemble_out([s.grid for s in solvers])
        return {"kind": "ensemble", "solvers": solvers, "ensemble": gea.Ensemble(solvers, stream=stream),
                "fields": fields, "out": outs, "flat": flat, "steps": case["steps"]}
    r, c, ax, az, theta = _network_inputs(case, seed)
    net = gea.Net(case["n"], case["h"], case["w"], relu=False, stream=stream)
    net.set_params(theta)
    return {"kind": "network", "net": net, "r": r, "c": c, "ax": ax, "az": az, "y": torch.empty_like(r),
            "dy": torch.empty_like(r), "grad": _empty(gea.net_param_count(), torch.float32)}


def run(state):
    if state["kind"] == "step":
        s = state["solver"]
        s.set_conservative(state["fields"])
        s.step(state["steps"])
        return s.get_state(state["out"]) if isinstance(s, gea.Solver3D) else s.get_full(state["out"])
    if state["kind"] == "ensemble":
        for s, f in zip(state["solvers"], state["fields"]):
            s.set_conservative(f)
        state["ensemble"].step(state["steps"])
        for s, o in zip(state["solvers"], state["out"]):
            s.get_full(o)
        return state["flat"]
    net = state["net"]
    net.forward(state["r"], state["y"])
    loss = net.energy(state["c"], state["ax"], state["az"], state["dy"])
    net.backward(state["dy"], state["grad"])
    return {"y": state["y"], "loss": loss, "dy": state["dy"], "grad": state["grad"]}


def work(case):
    """Bytes: the fields a call takes and returns. Flops per cell and step: each stage of Section 3 once on its
    stencils (one momentum and one enthalpy sweep per decade and a half of the solves' tolerance, one pressure
    operator application per decade)."""
    if case["kind"] == "network":
        n, h, w = case["n"], case["h"], case["w"]
        # multiply-adds of the forward layers per finest pixel, by level (a quarter of the pixels each)
        macs = (9 * 16 + 9 * 256 * 3 + 16) + (9 * 32 * (16 + 32 + 32 + 16)) / 4 + (
            9 * 64 * (32 + 64 + 64) + 9 * 64 * 32) / 16 + 9 * 64 * 128 / 64
        return {"bytes": 4 * n * h * w * 6 + 8 * 221073, "flops": 6 * macs * n * h * w}
    if case["kind"] == "step3d":
        cells, fields, flops = case["nx"] * case["ny"] * case["nz"], 5 + 7, 1100
    elif case["kind"] == "ensemble":
        cells, fields, flops = sum(n * n for n in _member_sizes(case)), 4 + 10, 700
    else:
        cells, fields, flops = case["nx"] * case["nz"], 4 + 10, 700
    return {"bytes": 8 * fields * cells, "flops": flops * cells * case["steps"]}


# ---- the same in plain torch, 64 bits ----

class _Box:
    """Stencils of Section 3 on a box of cells, arrays over z, (y,) x; direction 0 is x, the last one z."""

    def __init__(self, sizes, lengths, c):
        self.c, self.nd = c, len(sizes)
        self.n, self.h = sizes, [length / n for length, n in zip(lengths, sizes)]
        self.vol = math.prod(self.h)
        self.dims = [self.nd - 1 - d for d in range(self.nd)]
        self.gz = c.g * _axis(sizes[-1], lengths[-1], 0, self.nd)
        faces = c.g * torch.arange(1, sizes[-1], dtype=torch.float64, device=DEVICE) * self.h[-1]
        self.gzf = faces.reshape([-1] + [1] * (self.nd - 1))

    def cut(self, X, d, lo, hi):
        """X[lo : size + hi] along direction d."""
        return X.narrow(self.dims[d], lo, X.shape[self.dims[d]] + hi - lo)

    def ghosts(self, X, d, rule):
        """X with one ghost layer on both sides in direction d: "odd", "even", or "h" (dh/dz = -g)."""
        lo, hi = self.cut(X, d, 0, 1 - X.shape[self.dims[d]]), self.cut(X, d, X.shape[self.dims[d]] - 1, 0)
        if rule == "odd":
            lo, hi = -lo, -hi
        elif rule == "h":
            lo, hi = lo + self.c.g * self.h[d], hi - self.c.g * self.h[d]
        return torch.cat([lo, X, hi], self.dims[d])

    def grow(self, F, d):
        """Values on the inner faces of direction d with zeros on the walls."""
        zero = torch.zeros_like(self.cut(F, d, 0, 1 - F.shape[self.dims[d]]))
        return torch.cat([zero, F, zero], self.dims[d])

    def out(self, F, d):
        """Difference of a field on all faces of direction d."""
        return self.cut(F, d, 1, 0) - self.cut(F, d, 0, -1)

    def area(self, d):
        return self.vol / self.h[d]

    def diff(self, X, d):
        return self.cut(X, d, 1, 0) - self.cut(X, d, 0, -1)

    def mean(self, X, d):
        return 0.5 * (self.cut(X, d, 1, 0) + self.cut(X, d, 0, -1))

    def convect(self, phi, X, rules):
        total = 0.0
        for d in range(self.nd):
            G = self.ghosts(X, d, rules[d])
            face = (7.0 * (self.cut(G, d, 1, -2) + self.cut(G, d, 2, -1)) - self.cut(G, d, 0, -3)
                    - self.cut(G, d, 3, 0)) / 12.0
            total = total + self.out(phi[d] * self.grow(face, d), d)
        return total / self.vol

    def diffuse(self, mu, X, rules):
        total = 0.0
        for d in range(self.nd):
            grad = self.diff(self.ghosts(X, d, rules[d]), d) / self.h[d]
            m = mu if isinstance(mu, float) else self.mean(self.ghosts(mu, d, "even"), d)
            total = total + self.out(m * grad, d) / self.h[d]
        return total

    def force(self, pp, rho, d):
        """p' and buoyancy difference across the inner faces of direction d, over the spacing."""
        gz = self.gzf if d == self.nd - 1 else self.gz
        return (self.diff(pp, d) - gz * self.diff(rho, d)) / self.h[d]

    def to_cells(self, F, d):
        return self.mean(self.grow(F, d), d)


def _jacobi(op, diagonal, b, x):
    size = b.norm()
    for _ in range(60):
        r = b - op(x)
        x = x + r / diagonal
        if r.norm() <= 1e-15 * size:
            break
    return x


def _conjugate_gradients(op, diagonal, r, size):
    """The solution of op(x) = r from zero, to a residual of 1e-18 of `size`."""
    x = torch.zeros_like(r)
    z = r / diagonal
    p, rz = z.clone(), (r * z).sum()
    for k in range(3000):
        if k % 4 == 0 and r.norm() <= 1e-18 * size:
            break
        q = op(p)
        alpha = rz / (p * q).sum()
        x += alpha * p
        r = r - alpha * q
        z = r / diagonal
        rz, old = (r * z).sum(), rz
        p = z + (rz / old) * p
    return x


def _exact_steps(sizes, lengths, c, f, steps):
    """Steps of Section 3 from conservative fields: continuity and implicit momentum predictor, implicit enthalpy,
    equation of state, PISO correctors with the Helmholtz pressure equation."""
    B = _Box(sizes, lengths, c)
    nd, dt, z = B.nd, c.dt, B.nd - 1
    names = ("rhou", "rhow") if nd == 2 else ("rhou", "rhov", "rhow")
    rules = [["odd" if d == e else "even" for e in range(nd)] for d in range(nd)]
    even, enthalpy = ["even"] * nd, ["even"] * z + ["h"]
    rho = f["rho"]
    u = [f[k] / rho for k in names]
    T = (f["rhoe"] / rho - 0.5 * sum(v * v for v in u) - B.gz) / c.cv
    h, p = c.cp * T, rho * c.R * T
    pp, pold = p + rho * B.gz, p
    phi = [B.grow(B.mean(f[k], d) * B.area(d), d) for d, k in enumerate(names)]
    for _ in range(steps):
        mu = c.mu
        if c.cs > 0.0:
            grads = [[0.5 * (B.cut(B.ghosts(u[a], d, rules[a][d]), d, 2, 0)
                             - B.cut(B.ghosts(u[a], d, rules[a][d]), d, 0, -2)) / B.h[d] for d in range(nd)]
                     for a in range(nd)]
            s2 = sum(0.5 * (grads[a][d] + grads[d][a]) ** 2 for a in range(nd) for d in range(nd))
            mu = mu + rho * (c.cs * B.vol ** (1.0 / nd)) ** 2 * torch.sqrt(s2)
            del grads, s2
        div = sum(B.out(phi[d], d) for d in range(nd)) / B.vol
        rho1 = rho - dt * div
        mu_diag = sum(2.0 * mu / B.h[d] ** 2 for d in range(nd))   # any diagonal near the operator's will do
        diagonal = rho1 / dt + (7.0 / 12.0) * div + mu_diag

        def transport(X, rule, m):
            return rho1 / dt * X + B.convect(phi, X, rule) - B.diffuse(m, X, rule)
        u1 = []
        for d in range(nd):
            b = rho * u[d] / dt - B.to_cells(B.force(pp, rho, d), d)
            u1.append(_jacobi(lambda X, d=d: transport(X, rules[d], mu), diagonal, b, u[d]))
        K, K1 = 0.5 * sum(v * v for v in u), 0.5 * sum(v * v for v in u1)
        b = (rho * h + rho * K - pold) / dt - rho1 * K1 / dt - B.convect(phi, K1, even) + p / dt - rho1 * c.g * u1[z]
        h1 = _jacobi(lambda X: transport(X, enthalpy, mu if c.Pr == 1.0 else mu / c.Pr), diagonal, b, h)
        del K, K1, b, mu_diag, diagonal
        T1 = T + (h1 - h) / c.cp
        psi = 1.0 / (c.R * T1)
        rho2 = p * psi
        D = [dt * B.mean(rho2, d) / B.mean(rho1, d) for d in range(nd)]

        def helmholtz(X):
            return psi / dt * X - sum(B.out(B.grow(D[d] * B.diff(X, d), d), d) / B.h[d] ** 2 for d in range(nd))
        diag = psi / dt + sum(2.0 * B.to_cells(D[d], d) / B.h[d] ** 2 for d in range(nd))
        U, x = u1, pp
        for _ in range(c.n_corr):
            H = [rho * u[d] / dt + rho1 / dt * U[d] - transport(U[d], rules[d], mu) for d in range(nd)]
            b = (rho + psi * rho2 * B.gz) / dt
            for d in range(nd):
                gz = B.gzf if d == z else B.gz
                flux = D[d] * (B.mean(H[d], d) + gz * B.diff(rho2, d) / B.h[d])
                b = b - B.out(B.grow(flux, d), d) / B.h[d]
            x = x + _conjugate_gradients(helmholtz, diag, b - helmholtz(x), b.norm())
            G = [B.force(x, rho2, d) for d in range(nd)]
            new_phi = [B.grow(D[d] * (B.mean(H[d], d) - G[d]), d) * B.area(d) for d in range(nd)]
            U = [dt / rho1 * (H[d] - B.to_cells(G[d], d)) for d in range(nd)]
            del b, H, G
        phi, u, T, h, pold, pp = new_phi, U, T1, h1, p, x
        p = pp - rho2 * B.gz
        rho = p * psi
    state = {"rho": rho, "T": T, "h": h, "p": p, "pp": pp, "pold": pold}
    state.update(zip(("u", "w") if nd == 2 else ("u", "v", "w"), u))
    if nd == 2:
        state.update(phix=phi[0], phiz=phi[1])
    return state


def _exact_network(case, seed):
    r, c, ax, az, theta = _network_inputs(case, seed)
    theta = torch.tensor(theta, dtype=torch.float64, device=DEVICE, requires_grad=True)
    r, c, ax, az = (v.double() for v in (r, c, ax, az))
    channels = [(1, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 64), (64, 64), (64, 64), (64, 32),
                (32, 32), (32, 16), (16, 16), (16, 16), (16, 1)]
    layers, at = [], 0
    for i, (ci, co) in enumerate(channels):
        k = 1 if i == 14 else 3
        wt = theta[at:at + co * k * k * ci].reshape(co, k, k, ci).permute(0, 3, 1, 2)
        at += co * k * k * ci
        layers.append((wt, theta[at:at + co], k // 2))
        at += co
    F = torch.nn.functional

    def conv(i, x):
        return F.conv2d(x, layers[i][0], layers[i][1], padding=layers[i][2])

    def up(x):
        return F.interpolate(x, scale_factor=2, mode="nearest")
    x = (r / r.square().mean((1, 2), keepdim=True).sqrt())[:, None]
    e0 = conv(1, conv(0, x))
    e1 = conv(3, conv(2, F.avg_pool2d(e0, 2)))
    e2 = conv(5, conv(4, F.avg_pool2d(e1, 2)))
    e3 = conv(7, conv(6, F.avg_pool2d(e2, 2)))
    d2 = conv(9, conv(8, e2 + up(e3)))
    d1 = conv(11, conv(10, e1 + up(d2)))
    y = conv(14, conv(13, conv(12, e0 + up(d1))))[:, 0]
    v = y.detach()
    Av = c * v
    fx, fz = ax[:, :, 1:-1] * (v[:, :, 1:] - v[:, :, :-1]), az[:, 1:-1] * (v[:, 1:] - v[:, :-1])
    Av[:, :, :-1] -= fx
    Av[:, :, 1:] += fx
    Av[:, :-1] -= fz
    Av[:, 1:] += fz
    Av = Av / c.mean((1, 2), keepdim=True)
    n, hh, ww = r.shape
    dy = (Av - x[:, 0]) / (n * hh * ww)
    loss = ((0.5 * v * Av - v * x[:, 0]).sum() / (n * hh * ww)).item()
    y.backward(dy)
    return {"y": v, "loss": loss, "dy": dy, "grad": theta.grad}


def exact(case, seed):
    if case["kind"] == "network":
        return _exact_network(case, seed)
    if case["kind"] == "step3d":
        grid, c, f = _step3d_inputs(case, seed)
        got = _exact_steps((grid.nx, grid.ny, grid.nz), (grid.lx, grid.ly, grid.lz), c, f, case["steps"])
        return {k: got[k] for k in gea.STATE3_FIELDS}
    if case["kind"] == "step2d":
        grid, c, f = _step2d_inputs(case, case["nx"], case["nz"], seed)
        got = _exact_steps((grid.nx, grid.nz), (grid.lx, grid.lz), c, f, case["steps"])
        return {k: got[k] for k in gea.FULL_FIELDS[:-1]}
    parts = {k: [] for k in gea.FULL_FIELDS[:-1]}
    for m, n in enumerate(_member_sizes(case)):
        grid, c, f = _step2d_inputs(case, n, n, 1000 * seed + m)
        got = _exact_steps((n, n), (grid.lx, grid.lz), c, f, case["steps"])
        for k in parts:
            parts[k].append(got[k].reshape(-1))
    return {k: torch.cat(v) for k, v in parts.items()}
