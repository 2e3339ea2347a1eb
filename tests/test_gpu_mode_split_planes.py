"""FP64 mode sums as split integer products: every z plane keeps its own accuracy,
whatever its 16-plane tile holds, and the sums keep their last digits."""
import numpy as np
import pytest
import torch

from inputs.bunches import Geometry, Grid
from test_gpu_mode_split import make

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


def sinpi(v):
    """sin(pi v) of the FP64 number v, rounded once."""
    v = v.astype(LD)
    r = v - 2 * np.round(v / 2)
    pi = LD(np.pi) + LD(1.2246467991473532e-16)
    return np.sin(pi * r).astype(np.float64)


def sines(modes, origin, h, rows, length):
    """The solver's tables: sin(pi mode (origin + row h) / length), the argument's
    node rounded once (a fused multiply-add)."""
    x = (LD(origin) + np.arange(rows).astype(LD) * LD(h)).astype(np.float64)
    return sinpi(modes[:, None].astype(np.float64) * x[None, :] / length)


def tables(s):
    geom, grid = s.geometry, s.grid
    mx, mxp, myp, fold, xb = s.mode_layout()
    n = np.array([2 * q + 1 if q < myp // 2 else 2 * (q - myp // 2) + 2 for q in range(myp)]) if fold \
        else np.arange(1, myp + 1)
    m = np.arange(1, mxp + 1)
    sx = sines(m, geom.x0, grid.hx, grid.nx, geom.a) * (m <= geom.modes_m)[:, None]
    sy = sines(n, geom.y0, grid.hy, grid.ny, geom.b) * (n <= geom.modes_n)[:, None]
    return torch.tensor(sx).cuda(), torch.tensor(sy).cuda()


def project(sx, sy, rho):
    p = torch.matmul(sy, rho)
    return torch.matmul(sx, p.reshape(len(rho), -1)).reshape(-1, rho.shape[2])


def back(sx, sy, psi, nz):
    b = torch.matmul(sx.T, psi.reshape(len(sx), -1)).reshape(sx.shape[1], len(sy), nz)
    return torch.matmul(sy.T, b)


MESHES = [
    ("centred", 16, 16, 32, (20, 20)),
    ("centred", 48, 144, 64, (5, 7)),           # 72 pairs: a second run of 8
    ("wall", 80, 272, 32, (20, 21)),            # 136 pairs, three runs
    ("window", 112, 80, 32, (24, 28)),
    ("centred", 16, 32, 32, (32, 16)),
    ("centred", 1024, 16, 512, (20, 20)),       # four slabs of z
]


# Every value within 16 u per term of each of the two sums, in units of the
# largest value of its own z plane.
@pytest.mark.parametrize("kind,nx,ny,nz,modes", MESHES)
def test_planes_keep_their_own_accuracy(kind, nx, ny, nz, modes):
    s = make(kind, nx, ny, nz, modes)
    sx, sy = tables(s)
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    scale = torch.exp2(torch.randint(-60, 60, (nz,), device="cuda", generator=g).double())
    rho = (torch.rand(nx, ny, nz, **f) - 0.3) * scale
    part, psi = s.mode_buffers()
    s.stage_modes(0, rho, part)
    assert ((part.sum(0) - project(sx, sy, rho)).abs() <= 16 * U * nx * ny * scale).all()
    psi.copy_((torch.rand(psi.shape, **f) - 0.5) * scale)
    phi = s.empty()
    s.stage_modes(2, psi, phi)
    assert ((phi - back(sx, sy, psi, nz)).abs() <= 16 * U * len(psi) * scale).all()


# Values of mean zero, in the norm: N terms below 1/2 with independent errors, each
# below 1 u from the two tables, the half-transformed field, the cut digits and the
# result, and below 1.5 u from the reference's own sums (their partial sums grow as
# a random walk): 4 u sqrt(N) in all.  (The least weight of digit products left out
# is an error of about 200 u sqrt(N).)
@pytest.mark.parametrize("kind,nx,ny,nz,modes", MESHES)
def test_sums_keep_their_last_digits(kind, nx, ny, nz, modes):
    s = make(kind, nx, ny, nz, modes)
    sx, sy = tables(s)
    g = torch.Generator(device="cuda").manual_seed(7 + nx + ny)
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    rho = torch.rand(nx, ny, nz, **f) - 0.5
    part, psi = s.mode_buffers()
    s.stage_modes(0, rho, part)
    err = part.sum(0) - project(sx, sy, rho)
    assert err.square().mean().sqrt() <= 4 * U * (nx * ny) ** 0.5
    psi.copy_(torch.rand(psi.shape, **f) - 0.5)
    phi = s.empty()
    s.stage_modes(2, psi, phi)
    err = phi - back(sx, sy, psi, nz)
    assert err.square().mean().sqrt() <= 4 * U * len(psi) ** 0.5


def banded(kind, nb):
    from paper_1111_4971_gb300 import PipeSolver
    a, b, nx, ny, nz = 1.3, 1.0, 32, 48, 64
    geom = Geometry(a, b, 0.0, 0.0, 9, 11) if kind == "wall" else Geometry(a, b, a / nx / 2, b / ny / 2, 9, 11)
    s = PipeSolver(geom, Grid(nx, ny, nz, a / nx, b / ny, 0.05), igf=True, dtype=torch.float64, banded=nb)
    s.set_plan(t_kind=3)
    return s


@pytest.mark.parametrize("kind", ["centred", "wall"])
def test_banded_planes_are_independent(kind):
    """With no neighbours a plane's potential is its own density's: bit for bit what
    it is when the planes beside it are 2^80 larger or hold values that are not
    finite, which reach their own planes and as many neighbours as the band has."""
    g = torch.Generator(device="cuda").manual_seed(3)
    for nb in (0, 1):
        s = banded(kind, nb)
        rho = torch.rand(32, 48, 64, dtype=torch.float64, device="cuda", generator=g) - 0.3
        alone = rho.clone()
        alone[..., 20:23] = 0.0
        other = rho.clone()
        other[..., 20:23] *= 2.0 ** 80
        far = [k for k in range(64) if not 20 - nb <= k <= 22 + nb]
        want = s.solve(alone)
        assert torch.equal(s.solve(other)[..., far], want[..., far])
        for bad in (float("inf"), float("nan")):
            r = rho.clone()
            r[3, 0 if kind == "wall" else 5, 20] = bad
            phi = s.solve(r)
            hit = [k for k in range(64) if abs(k - 20) <= nb]
            rest = [k for k in range(64) if abs(k - 20) > nb]
            assert not phi[..., hit].isfinite().any()
            assert torch.equal(phi[..., rest], s.solve(rho)[..., rest])
