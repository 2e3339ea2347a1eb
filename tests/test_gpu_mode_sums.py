"""FP32 projection of the mode-space form against the plain FP64 sums where the
x-mode sums take their slots two at a time: slots missing in the last pair, four
and eight warps, x modes at the edge of the one-by-one form, repeated x blocks."""
import numpy as np
import pytest
import torch

from inputs.bunches import Geometry, Grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


# One sum has at most ny + nx additions and two rounded tables: every value is
# within (ny + nx + 4) u of the sum of |Sx Sy rho| over the mesh.
@pytest.mark.parametrize("kind,nx,ny,nz,modes", [
    ("centred", 16, 16, 64, (20, 8)),           # 4 warps, 8 slots: every pair full
    ("centred", 32, 16, 32, (17, 12)),          # 4 warps, 12 slots: one left over for each
    ("centred", 128, 16, 512, (20, 20)),        # 8 warps, 20 slots: for half of them
    ("centred", 128, 16, 512, (4, 12)),         # the second of a pair missing for half
    ("centred", 128, 16, 512, (21, 24)),        # one by one
    ("wall", 64, 32, 32, (20, 16)),
    ("window", 48, 80, 64, (20, 24)),
    ("window", 48, 80, 64, (1, 32)),
    ("centred", 512, 16, 64, (20, 20)),         # several x blocks a CTA
])
def test_projection_against_plain_sums(kind, nx, ny, nz, modes):
    from paper_1111_4971_gb300 import PipeSolver
    a, b = 1.3, 1.0
    if kind == "window":
        geom, hx, hy = Geometry(a, b, 0.13, 0.11, *modes), 0.5 * a / nx, 0.6 * b / ny
    elif kind == "wall":
        geom, hx, hy = Geometry(a, b, 0.0, 0.0, *modes), a / nx, b / ny
    else:
        geom, hx, hy = Geometry(a, b, a / nx / 2, b / ny / 2, *modes), a / nx, b / ny
    s = PipeSolver(geom, Grid(nx, ny, nz, hx, hy, 0.05), igf=True, dtype=torch.float32)
    s.set_plan(t_kind=3)
    mx, mxp, myp, fold, xb = s.mode_layout()
    m = np.arange(1, mxp + 1)
    n = np.array([2 * q + 1 if q < myp // 2 else 2 * (q - myp // 2) + 2 for q in range(myp)]) if fold \
        else np.arange(1, myp + 1)
    sx = np.sin(np.pi * m[:, None] * (geom.x0 + hx * np.arange(nx)) / a) * (m <= modes[0])[:, None]
    sy = np.sin(np.pi * n[:, None] * (geom.y0 + hy * np.arange(ny)) / b) * (n <= modes[1])[:, None]
    rho = np.random.default_rng(nx + ny).uniform(-0.3, 0.7, (nx, ny, nz)).astype(np.float32)
    part, psi = s.mode_buffers()
    part.fill_(float("nan"))
    s.stage_modes(0, torch.tensor(rho).cuda(), part)
    got = part.double().cpu().numpy().sum(axis=0).reshape(mxp, myp, nz)
    want = np.einsum("mx,xnz->mnz", sx, np.einsum("ny,xyz->xnz", sy, rho.astype(np.float64), optimize=True), optimize=True)
    bound = np.einsum("mx,xnz->mnz", abs(sx), np.einsum("ny,xyz->xnz", abs(sy), abs(rho).astype(np.float64), optimize=True),
                      optimize=True)
    assert (np.abs(got - want) <= (nx + ny + 4) * 2.0 ** -24 * bound + 1e-12).all()
