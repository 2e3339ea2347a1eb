"""FP64 mode sums as split integer products (projection and back-projection of
the mode-space form): against the plain sums at the sizes where the tiling can
go wrong, and over the exponent range."""
import numpy as np
import pytest
import torch

from inputs.bunches import Geometry, Grid

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


def make(kind, nx, ny, nz, modes):
    from paper_1111_4971_gb300 import PipeSolver
    a, b = 1.3, 1.0
    if kind == "window":
        geom, hx, hy = Geometry(a, b, 0.13, 0.11, *modes), 0.5 * a / nx, 0.6 * b / ny
    elif kind == "wall":
        geom, hx, hy = Geometry(a, b, 0.0, 0.0, *modes), a / nx, b / ny
    else:
        geom, hx, hy = Geometry(a, b, a / nx / 2, b / ny / 2, *modes), a / nx, b / ny
    s = PipeSolver(geom, Grid(nx, ny, nz, hx, hy, 0.05), igf=True, dtype=torch.float64)
    s.set_plan(t_kind=3)
    return s


def tables(s):
    geom, grid = s.geometry, s.grid
    mx, mxp, myp, fold, xb = s.mode_layout()
    n = np.array([2 * q + 1 if q < myp // 2 else 2 * (q - myp // 2) + 2 for q in range(myp)]) if fold \
        else np.arange(1, myp + 1)
    m = np.arange(1, mxp + 1)
    x = geom.x0 + grid.hx * np.arange(grid.nx)
    y = geom.y0 + grid.hy * np.arange(grid.ny)
    sx = np.sin(np.pi * m[:, None] * x / geom.a) * (m <= geom.modes_m)[:, None]
    sy = np.sin(np.pi * n[:, None] * y / geom.b) * (n <= geom.modes_n)[:, None]
    return torch.tensor(sx).cuda(), torch.tensor(sy).cuda()


def project(sx, sy, rho):
    p = torch.matmul(sy, rho)
    return torch.matmul(sx, p.reshape(len(rho), -1)).reshape(-1, rho.shape[2])


def back(sx, sy, psi, nz):
    b = torch.matmul(sx.T, psi.reshape(len(sx), -1)).reshape(sx.shape[1], len(sy), nz)
    return torch.matmul(sy.T, b)


# Error of one split sum over K terms below c in size: the cut of the data
# (2^-52 c), of the table (2^-54 c) and the dropped products (5 2^-54 c) a term,
# one rounding of the result: below 6 u K c.  The sine tables of the reference
# differ by up to 8 u (numpy's argument), the reference itself by u per term:
# together below 16 u per term of each of the two sums, in units of the largest
# value of a 16-value z tile.
@pytest.mark.parametrize("kind,nx,ny,nz,modes", [
    ("centred", 16, 16, 32, (20, 20)),          # fewer rows than a k step of pairs
    ("centred", 48, 144, 64, (5, 7)),           # 72 pairs: a second run of 8
    ("wall", 32, 16, 32, (24, 24)),
    ("wall", 80, 272, 32, (20, 21)),            # 136 pairs, three runs
    ("window", 16, 48, 64, (1, 1)),
    ("window", 112, 80, 32, (24, 28)),          # 32 y slots, 24 x slots
    ("centred", 16, 32, 32, (32, 16)),          # two k steps of x modes, 8-mode halves
    ("centred", 1024, 16, 512, (20, 20)),       # four slabs of z
])
def test_split_sums(kind, nx, ny, nz, modes):
    s = make(kind, nx, ny, nz, modes)
    sx, sy = tables(s)
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    rho = torch.rand(nx, ny, nz, dtype=torch.float64, device="cuda", generator=g) - 0.3
    rho *= torch.exp2(torch.randint(-30, 30, (1, 1, nz // 16), device="cuda", generator=g).double()).repeat_interleave(16, 2)
    part, psi = s.mode_buffers()
    s.stage_modes(0, rho, part)
    top = rho.abs().amax((0, 1)).reshape(-1, 16).amax(1).repeat_interleave(16)
    assert ((part.sum(0) - project(sx, sy, rho)).abs() <= 16 * U * nx * ny * top).all()
    psi.copy_(torch.rand(psi.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5)
    psi *= torch.exp2(torch.randint(-30, 30, (1, nz // 16), device="cuda", generator=g).double()).repeat_interleave(16, 1)
    phi = s.empty()
    s.stage_modes(2, psi, phi)
    top = psi.abs().amax(0).reshape(-1, 16).amax(1).repeat_interleave(16)
    assert ((phi - back(sx, sy, psi, nz)).abs() <= 16 * U * len(psi) * top).all()


@pytest.mark.parametrize("kind", ["centred", "wall", "window"])
def test_split_sums_over_the_exponent_range(kind):
    """A power of two in is the same power out, bit for bit, up to where results
    overflow or become subnormal; zeros give zeros; a value that is not finite
    leaves no finite value in its z tile."""
    s = make(kind, 32, 48, 32, (7, 9))
    g = torch.Generator(device="cuda").manual_seed(5)
    rho = torch.rand(32, 48, 32, dtype=torch.float64, device="cuda", generator=g) - 0.3
    part, psi = s.mode_buffers()

    def run(r):
        p = torch.empty_like(part)
        s.stage_modes(0, r, p)
        return p

    psi.copy_(torch.rand(psi.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5)

    def expand(v):
        phi = s.empty()
        s.stage_modes(2, v, phi)
        return phi

    p0, f0 = run(rho), expand(psi)
    for k in (-900, -40, 700, 1005):
        assert torch.equal(run(rho * 2.0 ** k), p0 * 2.0 ** k)
        assert torch.equal(expand(psi * 2.0 ** k), f0 * 2.0 ** k)
    # subnormal inputs are integers of 2^-1074: their sums to a unit of it, and to rounding
    tiny = torch.round(rho * 2.0 ** 40) * 2.0 ** -1000 * 2.0 ** -74
    want = run(torch.round(rho * 2.0 ** 40))
    assert ((run(tiny) * 2.0 ** 1000 * 2.0 ** 74 - want).abs() <= 32 * (1.0 + want.abs() * U) + 16 * U * 32 * 48 * 2.0 ** 40).all()
    assert (run(torch.zeros_like(rho)) == 0).all() and (expand(torch.zeros_like(psi)) == 0).all()
    for bad in (float("inf"), float("nan")):
        r = rho.clone()
        r[3, 0, 20] = bad
        p = run(r)
        assert p[..., 16:].isnan().all() and torch.equal(p[..., :16], p0[..., :16])
        v = psi.clone()
        v[1, 3] = bad
        f = expand(v)
        assert f[..., :16].isnan().all() and torch.equal(f[..., 16:], f0[..., 16:])
