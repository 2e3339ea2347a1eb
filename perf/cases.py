"""Workloads of the pipe-Poisson solver through its public Python entry points.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the handle(s) and the inputs a program holds before the call, on the GPU
    run(state)           one pass through the public entry points
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    what run() returns for these inputs, from plain 64-bit torch

A case is one mesh, one Green function, one dtype and one operation:

    op      solve    phi = A rho
            adjoint  rho' = A^T phi'
            pic      deposit macroparticles, solve, field E = -grad phi (a space-charge kick)
            grad     deposit, solve, W = 1/2 sum rho phi, and dW/d(positions) (beam optimisation)
            batch    many independent solves of mixed grids and aspect ratios in one call
    mesh    centred  cell centres, spanning the pipe
            wall     x0 = y0 = 0, spanning the pipe (the accuracy study's nodes)
            window   a transverse window of the pipe, off centre
    green   igf, ordinary, free (the free-space comparison solve)
    banded  -1 the full operator, else the neighbour planes kept on each side
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_1111_4971_gb300 import (CICDeposit, PipePoissonFunction, PipeSolver, field_energy,
                                   solve_batched)

DTYPES = {"f32": torch.float32, "f64": torch.float64}
BATCH_GRIDS = ((32, 64), (64, 128), (64, 256), (128, 512))      # (nx = ny, nz) of the mixed batch


def _case(op, nx, ny, nz, dtype, *, aspect=1.0, mesh="centred", green="igf", modes=20, banded=-1,
          particles=0, solves=0, **name):
    return dict(name, op=op, nx=nx, ny=ny, nz=nz, dtype=dtype, aspect=aspect, mesh=mesh, green=green,
                modes=modes, banded=banded, particles=particles, solves=solves)


def listed():
    return [
        # a small check-out mesh in full precision: all latency and launches
        _case("solve", 16, 16, 32, "f64", green="ordinary", name="solve16x16x32_f64"),
        # a Green function kept to 40 modes an axis, for beams with sharp transverse edges
        _case("solve", 64, 64, 256, "f32", aspect=2.0, modes=40, name="solve64x64x256_f32_modes40"),
        # one space-charge step of a tracking code on its usual mesh
        _case("pic", 64, 64, 256, "f32", aspect=2.0, particles=1 << 18, name="pic64x64x256_f32"),
        # a beam small against the pipe: a ragged window mesh beside the axis
        _case("adjoint", 48, 80, 512, "f32", aspect=1.5, mesh="window", name="window48x80x512_f32"),
        # the standard long-bunch solve, in both precisions
        _case("solve", 128, 128, 1024, "f32", name="solve128x128x1024_f32"),
        _case("solve", 128, 128, 1024, "f64", name="solve128x128x1024_f64"),
        # its banded reduction, for bunches long against the pipe
        _case("solve", 128, 128, 1024, "f32", banded=8, name="banded128x128x1024_f32"),
        # and the free-space solve it is compared with
        _case("solve", 128, 128, 1024, "f32", green="free", name="free128x128x1024_f32"),
        # gradients of the field energy with respect to a million macroparticles
        _case("grad", 128, 128, 512, "f32", particles=1 << 20, name="grad128x128x512_f32"),
        # an accuracy-study mesh with nodes on the wall
        _case("solve", 256, 256, 512, "f64", mesh="wall", name="wall256x256x512_f64"),
        # a parameter scan: 96 mixed solves in one call
        _case("batch", 128, 128, 512, "f32", solves=96, name="batch96_f32"),
        # the finest mesh in use
        _case("solve", 512, 512, 1024, "f32", name="solve512x512x1024_f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another mesh, aspect ratio and mode count of one of the listed kinds."""
    kind = rng.choice(["solve", "solve", "adjoint", "window", "wall", "banded", "free", "modes", "pic",
                       "grad", "batch"])
    dtype = rng.choice(["f32", "f32", "f64"])
    aspect = round(rng.uniform(1.0, 3.0), 3)
    nz = 1 << rng.randint(5, 10)
    side = 1 << rng.randint(4, 7)
    if kind == "batch":
        return _case("batch", 128, 128, 512, "f32", solves=_log_int(rng, 5, 96), aspect=aspect)
    if kind == "free":                       # meshes of the padded transforms: squares
        return _case("solve", side, side, nz, dtype, aspect=aspect, green="free")
    if kind == "modes":
        return _case("solve", side, side, nz, dtype, aspect=aspect, modes=rng.randint(33, 48))
    # sides in steps of 16, at most 2^24 nodes
    nx = 16 * _log_int(rng, 1, 20)
    ny = 16 * _log_int(rng, 1, 20)
    while nx * ny * nz > 1 << 24:
        nz //= 2
    modes = rng.choice([12, 16, 20, 20, 24])
    green = rng.choice(["igf", "igf", "ordinary"])
    if kind in ("pic", "grad"):
        return _case(kind, nx, ny, nz, dtype, aspect=aspect, modes=modes,
                     particles=_log_int(rng, 1 << 14, 1 << 20))
    if kind == "banded":
        return _case("solve", nx, ny, nz, dtype, aspect=aspect, green=green, modes=modes,
                     banded=_log_int(rng, 1, 17) - 1)
    mesh = {"window": "window", "wall": "wall"}.get(kind, rng.choice(["centred", "centred", "wall"]))
    op = "adjoint" if kind == "adjoint" else "solve"
    return _case(op, nx, ny, nz, dtype, aspect=aspect, mesh=mesh, green=green, modes=modes)


def _problem(case):
    """(geometry, grid) of a case: b = 1, a = aspect, the mesh 8 pipe heights long."""
    a, b = float(case["aspect"]), 1.0
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    hx, hy, hz = a / nx, b / ny, 8.0 / nz
    x0, y0 = hx / 2, hy / 2
    if case["mesh"] == "wall":
        x0 = y0 = 0.0
    elif case["mesh"] == "window":           # half the pipe's width, beside the axis
        hx, hy = 0.5 * a / nx, 0.5 * b / ny
        x0, y0 = 0.31 * a, 0.22 * b
    m = case["modes"]
    return (SimpleNamespace(a=a, b=b, x0=x0, y0=y0, modes_m=m, modes_n=m),
            SimpleNamespace(nx=nx, ny=ny, nz=nz, hx=hx, hy=hy, hz=hz))


def _solver(case):
    geom, grid = _problem(case)
    free = case["green"] == "free"
    return PipeSolver(geom, grid, igf=case["green"] == "igf", dtype=DTYPES[case["dtype"]], free_space=free,
                      banded=None if case["banded"] < 0 else case["banded"])


def _batch_cases(case):
    """The solves of a batch: a fixed mix of grids and aspect ratios for its size."""
    g = torch.Generator().manual_seed(1000 + case["solves"])
    out = []
    for _ in range(case["solves"]):
        n, nz = BATCH_GRIDS[int(torch.randint(len(BATCH_GRIDS), (1,), generator=g))]
        aspect = 1.0 + 2.0 * float(torch.rand(1, generator=g))
        out.append(dict(case, op="solve", nx=n, ny=n, nz=nz, aspect=aspect, solves=0))
    return out


def _bunch(case, g):
    """Centre and rms sizes of a bunch inside the mesh."""
    geom, grid = _problem(case)
    u = torch.rand(6, generator=g, device="cuda", dtype=torch.float64).tolist()
    lx, ly, lz = grid.nx * grid.hx, grid.ny * grid.hy, grid.nz * grid.hz
    centre = (geom.x0 + lx * (0.4 + 0.2 * u[0]), geom.y0 + ly * (0.4 + 0.2 * u[1]), lz * (0.45 + 0.1 * u[2]))
    sigma = (lx * (0.08 + 0.1 * u[3]), ly * (0.08 + 0.1 * u[4]), lz * (0.08 + 0.07 * u[5]))
    return centre, sigma


def _density(case, g):
    """A Gaussian bunch cut at three sigma, with a few per cent of shot noise."""
    geom, grid = _problem(case)
    centre, sigma = _bunch(case, g)
    f = dict(device="cuda", dtype=torch.float64)
    q = [((o + h * torch.arange(n, **f)) - c) / s for o, h, n, c, s in
         zip((geom.x0, geom.y0, 0.0), (grid.hx, grid.hy, grid.hz), (grid.nx, grid.ny, grid.nz), centre, sigma)]
    q2 = [(t * t).to(torch.float32) for t in q]
    r2 = q2[0][:, None, None] + q2[1][None, :, None] + q2[2][None, None, :]
    rho = torch.exp(-0.5 * r2)
    rho *= 1.0 + 0.05 * torch.randn(rho.shape, generator=g, device="cuda")
    rho.masked_fill_(r2 > 9.0, 0.0)
    rho /= (2 * math.pi) ** 1.5 * sigma[0] * sigma[1] * sigma[2]
    return rho.to(DTYPES[case["dtype"]])


def _particles(case, g):
    """Macroparticles of a Gaussian bunch drawn inside three sigma."""
    centre, sigma = _bunch(case, g)
    f = dict(device="cuda", dtype=torch.float64)
    xi = torch.randn(case["particles"], 3, generator=g, **f)
    r = xi.norm(dim=1, keepdim=True)
    xi *= torch.where(r > 3.0, 3.0 / r * torch.rand(r.shape, generator=g, **f), torch.ones_like(r))
    return (torch.tensor(centre, **f) + xi * torch.tensor(sigma, **f)).to(DTYPES[case["dtype"]]).contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def prepare(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "batch":
        cases = _batch_cases(case)
        solvers = [_solver(c) for c in cases]
        rhos = [_density(c, g) for c in cases]
        flat = torch.empty(sum(r.numel() for r in rhos), device="cuda")
        phis, at = [], 0
        for r in rhos:
            phis.append(flat[at:at + r.numel()].view(r.shape))
            at += r.numel()
        solve_batched(solvers, rhos, phis)   # the set's launch plan is chosen at its first call
        return dict(op=op, solvers=solvers, rhos=rhos, phis=phis, flat=flat)
    state = dict(op=op, solver=_solver(case))
    if op in ("pic", "grad"):
        state.update(xyz=_particles(case, g), charge=1.0 / case["particles"])
    else:
        state.update(rho=_density(case, g))
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        solve_batched(state["solvers"], state["rhos"], state["phis"])
        return state["flat"]
    solver = state["solver"]
    if op == "solve":
        return solver.solve(state["rho"])
    if op == "adjoint":
        return solver.adjoint(state["rho"])
    if op == "pic":
        rho = solver.cic_deposit(state["xyz"], state["charge"])
        phi = solver.solve(rho)
        return {"rho": rho, "phi": phi, "E": solver.electric_field(phi)}
    xyz = state["xyz"].detach().requires_grad_(True)
    rho = CICDeposit.apply(xyz, solver, state["charge"])
    phi = PipePoissonFunction.apply(rho, solver)
    energy = field_energy(rho, phi)
    (grad,) = torch.autograd.grad(energy, xyz)
    return {"energy": energy.detach(), "phi": phi.detach(), "grad": grad}


def work(case):
    if case["op"] == "batch":
        parts = [work(c) for c in _batch_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nodes, size, m = nx * ny * nz, 8 if case["dtype"] == "f64" else 4, case["modes"]
    particles = case["particles"]
    if case["green"] == "free":              # two padded real transforms
        flops = 2 * 2.5 * 8 * nodes * math.log2(8 * nodes)
    else:                                    # the mode sums along one axis, then the other, both ways;
        columns = m * m * nz                 # mirror images about a mid-plane share the first
        first = nodes * m if case["mesh"] == "centred" else 2 * nodes * m
        flops = 2 * (first + 2 * columns * min(nx, ny))
        # the recurrence or the band along z
        flops += columns * (8 if case["banded"] < 0 else 2 * (2 * case["banded"] + 1))
    if case["op"] == "pic":                  # positions in; density, potential and field out
        return {"bytes": (3 * particles + 5 * nodes) * size, "flops": flops + 40 * particles + 9 * nodes}
    if case["op"] == "grad":                 # positions in; potential and gradient out
        return {"bytes": (6 * particles + nodes) * size, "flops": 2 * flops + 120 * particles + 2 * nodes}
    return {"bytes": 2 * nodes * size, "flops": flops}


# -- the same in 64-bit torch ------------------------------------------------

def _lag_kernel(case, kappa, hz, nz):
    """z kernel of each mode at the lags 0..nz-1: exp(-kappa z), or its integral over a cell's hat."""
    d = torch.arange(nz, device="cuda", dtype=torch.float64)
    k = kappa[..., None]
    if case["green"] == "ordinary":
        f = torch.exp(-k * d * hz)
    else:
        t = k * hz
        f = (2 * torch.sinh(t / 2) / t) ** 2 * torch.exp(-t * d)
        f[..., 0] = 2 * (t[..., 0] + torch.expm1(-t[..., 0])) / t[..., 0] ** 2
    if case["banded"] >= 0:
        f[..., case["banded"] + 1:] = 0.0
    return f


def _exact_pipe(case, rho):
    geom, grid = _problem(case)
    f = dict(device="cuda", dtype=torch.float64)
    m = torch.arange(1, case["modes"] + 1, **f)
    sx = torch.sin(torch.outer(m, math.pi / geom.a * (geom.x0 + grid.hx * torch.arange(grid.nx, **f))))
    sy = torch.sin(torch.outer(m, math.pi / geom.b * (geom.y0 + grid.hy * torch.arange(grid.ny, **f))))
    kappa = math.pi * torch.sqrt((m[:, None] / geom.a) ** 2 + (m[None, :] / geom.b) ** 2)
    nz = grid.nz
    p = torch.matmul(sy, rho)                                               # [nx][n][nz]
    p = torch.matmul(sx, p.reshape(grid.nx, -1)).reshape(len(m), len(m), nz)  # [m][n][nz]
    lag = _lag_kernel(case, kappa, grid.hz, nz)
    ext = torch.cat([lag, torch.zeros_like(lag[..., :1]), lag[..., 1:].flip(-1)], -1)
    psi = torch.fft.irfft(torch.fft.rfft(p, 2 * nz) * torch.fft.rfft(ext), 2 * nz)[..., :nz]
    psi = psi * (grid.hx * grid.hy * grid.hz * 8 * math.pi / (geom.a * geom.b) / kappa)[..., None]
    b = torch.matmul(sx.T, psi.reshape(len(m), -1)).reshape(grid.nx, len(m), nz)
    return torch.matmul(sy.T, b)


def _exact_free(case, rho):
    _, grid = _problem(case)
    f = dict(device="cuda", dtype=torch.float64)
    r2 = 0.0
    for axis, (n, h) in enumerate(((grid.nx, grid.hx), (grid.ny, grid.hy), (grid.nz, grid.hz))):
        i = torch.arange(2 * n, **f)
        shape = [1, 1, 1]
        shape[axis] = 2 * n
        r2 = r2 + (torch.minimum(i, 2 * n - i) * h).reshape(shape) ** 2
    r2[0, 0, 0] = min(grid.hx, grid.hy, grid.hz) ** 2
    s = r2.shape
    g = torch.fft.rfftn(r2.rsqrt_())
    g *= torch.fft.rfftn(rho, s)
    phi = torch.fft.irfftn(g, s)[:grid.nx, :grid.ny, :grid.nz]
    return (phi * (grid.hx * grid.hy * grid.hz)).contiguous()


def _exact_solve(case, rho):
    return _exact_free(case, rho) if case["green"] == "free" else _exact_pipe(case, rho)


def _corners(case, xyz):
    """For each of a cell's eight nodes: flat index, inside the mesh, weights and slopes by axis."""
    geom, grid = _problem(case)
    f = dict(device="cuda", dtype=torch.float64)
    h = torch.tensor([grid.hx, grid.hy, grid.hz], **f)
    n = torch.tensor([grid.nx, grid.ny, grid.nz], device="cuda")
    u = (xyz - torch.tensor([geom.x0, geom.y0, 0.0], **f)) / h
    i0 = torch.floor(u)
    d = u - i0
    for corner in range(8):
        s = torch.tensor([corner >> 2 & 1, corner >> 1 & 1, corner & 1], device="cuda")
        w = torch.where(s == 1, d, 1 - d)
        slope = torch.where(s == 1, 1.0, -1.0) / h
        i = i0.long() + s
        ok = ((i >= 0) & (i < n)).all(1)
        i = torch.minimum(i.clamp(min=0), n - 1)
        yield (i[:, 0] * grid.ny + i[:, 1]) * grid.nz + i[:, 2], ok, w, slope


def _exact_deposit(case, xyz, charge):
    _, grid = _problem(case)
    rho = torch.zeros(grid.nx * grid.ny * grid.nz, device="cuda", dtype=torch.float64)
    for at, ok, w, _ in _corners(case, xyz):
        rho.index_add_(0, at, w.prod(1) * ok)
    return (rho * (charge / (grid.hx * grid.hy * grid.hz))).reshape(grid.nx, grid.ny, grid.nz)


def _exact_position_grad(case, xyz, charge, field):
    _, grid = _problem(case)
    out = torch.zeros_like(xyz)
    for at, ok, w, slope in _corners(case, xyz):
        v = field.reshape(-1)[at] * ok
        for axis in range(3):
            others = [k for k in range(3) if k != axis]
            out[:, axis] += v * slope[axis] * w[:, others[0]] * w[:, others[1]]
    return out * (charge / (grid.hx * grid.hy * grid.hz))


def exact(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "batch":
        cases = _batch_cases(case)
        return torch.cat([_exact_solve(c, _density(c, g).double()).reshape(-1) for c in cases])
    if op in ("solve", "adjoint"):           # G(r, r') = G(r', r): the operator is symmetric
        return _exact_solve(case, _density(case, g).double())
    _, grid = _problem(case)
    xyz, charge = _particles(case, g).double(), 1.0 / case["particles"]
    rho = _exact_deposit(case, xyz, charge)
    phi = _exact_solve(case, rho)
    if op == "pic":
        E = torch.stack(torch.gradient(phi, spacing=(grid.hx, grid.hy, grid.hz), edge_order=2)).neg()
        return {"rho": rho, "phi": phi, "E": E}
    return {"energy": 0.5 * (rho * phi).sum(), "phi": phi,
            "grad": _exact_position_grad(case, xyz, charge, phi)}
