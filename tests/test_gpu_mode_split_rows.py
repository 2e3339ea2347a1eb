"""FP64 mode sums as split integer products next to the pipe's walls, where every
sine of a table row is small: the sums keep their accuracy relative to the row."""
import numpy as np
import pytest
import torch

from inputs.bunches import Geometry, Grid
from test_gpu_mode_split import make
from test_gpu_mode_split_planes import back, project, sinpi, tables

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


def rows(t):
    """The largest sine of each mesh row."""
    return t.abs().amax(0)


# A row's digits are cut 2^-54 below a power of two at most twice its largest sine
# c, the data's 2^-52 below the largest value: with the dropped products (5 2^-54)
# below 12 u c a term of each sum; the tables of the reference and its own sums add
# 3 u: 16 u per term, in units of c and of the largest value.  (Cut 2^-54 below 1,
# a term is off by u / 2c: 100 u c at c = 0.005.)
@pytest.mark.parametrize("kind,nx,ny,nz,modes", [
    ("centred", 16, 1024, 32, (3, 3)),          # c = 0.0046 in the first row, folded
    ("centred", 1024, 16, 32, (2, 5)),          # along x: both ends
    ("wall", 512, 512, 32, (3, 4)),             # first rows on the wall
    ("window", 64, 48, 64, (7, 9)),
])
def test_rows_next_to_a_wall(kind, nx, ny, nz, modes):
    s = make(kind, nx, ny, nz, modes)
    sx, sy = tables(s)
    cx, cy = rows(sx), rows(sy)
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    part, psi = s.mode_buffers()
    psi.copy_(torch.rand(psi.shape, **f) - 0.5)
    phi = s.empty()
    s.stage_modes(2, psi, phi)
    bound = 16 * U * len(psi) * cx[:, None, None] * cy[None, :, None]
    assert ((phi - back(sx, sy, psi, nz)).abs() <= bound).all()
    # a density in single rows, each plane in its own
    rho = s.empty().zero_()
    ix = torch.tensor([0, 1, nx - 1, nx // 3]).repeat(nz // 4).cuda()
    jy = torch.tensor([0, 1, ny - 1, ny // 3, 2]).repeat(nz)[:nz].cuda()
    k = torch.arange(nz).cuda()
    rho[ix, jy, k] = torch.rand(nz, **f) + 0.5
    s.stage_modes(0, rho, part)
    assert ((part.sum(0) - project(sx, sy, rho)).abs() <= 16 * U * 2 * cx[ix] * cy[jy] * rho[ix, jy, k]).all()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_density_on_the_wall_is_not_felt(dtype):
    """Rows on the wall have zero sines: whatever finite density they hold, the
    potential is bit for bit that of none."""
    from paper_1111_4971_gb300 import PipeSolver
    a, b, nx, ny, nz = 1.3, 1.0, 32, 48, 64
    s = PipeSolver(Geometry(a, b, 0.0, 0.0, 9, 11), Grid(nx, ny, nz, a / nx, b / ny, 0.05), igf=True, dtype=dtype)
    s.set_plan(t_kind=3)
    g = torch.Generator(device="cuda").manual_seed(1)
    rho = torch.rand(nx, ny, nz, dtype=dtype, device="cuda", generator=g) - 0.3
    rho[0] = 0.0
    rho[:, 0] = 0.0
    want = s.solve(rho)
    assert want.abs().max() > 0
    for scale in (1.0, 2.0 ** 60):
        r = rho.clone()
        r[0] = scale
        r[:, 0] = -scale
        assert torch.equal(s.solve(r), want)


def test_tables_that_sum_fewer_rows_at_a_time():
    """A window so narrow that a mode's sines agree in every row and all their
    digits are large: 64 such rows pass what the accumulators hold exactly, so the
    contraction over y takes 32 at a time."""
    from paper_1111_4971_gb300 import PipeSolver
    n = np.arange(1, 33)

    def digits(t):
        x = int(np.rint(np.ldexp(t, 53 + max(0, -int(np.frexp(abs(t))[1])))))
        out = []
        for _ in range(5):
            out.append((x + 256) % 512 - 256)
            x = (x - out[-1]) // 512
        return np.abs([x] + out[::-1])

    def heaviest(y0):
        return max(digits(float(t))[:5].sum() for t in sinpi(n.astype(np.float64) * y0))

    y0 = max((k / 997 for k in range(100, 400)), key=heaviest)
    assert 64 * 256 * heaviest(y0) > 1.02 * 2 ** 24
    nx, ny, nz = 16, 80, 32
    s = PipeSolver(Geometry(1.3, 1.0, 0.05, y0, 6, 32), Grid(nx, ny, nz, 0.07, 1e-19, 0.05), igf=True, dtype=torch.float64)
    s.set_plan(t_kind=3)
    sx, sy = tables(s)
    g = torch.Generator(device="cuda").manual_seed(2)
    rho = torch.rand(nx, ny, nz, dtype=torch.float64, device="cuda", generator=g) - 0.3
    part, psi = s.mode_buffers()
    s.stage_modes(0, rho, part)
    assert ((part.sum(0) - project(sx, sy, rho)).abs() <= 16 * U * nx * ny).all()
