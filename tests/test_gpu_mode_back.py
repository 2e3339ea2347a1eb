"""FP32 back-projection of the mode-space form against the plain FP64 sums, in the
norm: its sums run from the small terms to the large ones, so that few roundings
are as large as the result's own."""
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


# Mode columns that fall as a potential's do.  Roundings of the result's own size:
# two tables, B, the last additions of O and of E, O + E; each is about 0.4 u of
# its value in the norm, sqrt(6) 0.4 u = 1 u together, and those before them are
# a quarter of that at most: 1.25 u.  (The sums taken from the first mode up have
# one such rounding per mode: emulated, 1.5 u at 8 modes, 2.3 to 3 u at 20 to 32.)
@pytest.mark.parametrize("kind,nx,ny,nz,modes", [
    ("centred", 32, 32, 64, (20, 20)),
    ("centred", 64, 48, 32, (32, 32)),
    ("centred", 16, 16, 32, (8, 7)),
    ("centred", 128, 64, 512, (20, 12)),        # 8 warps
    ("window", 48, 80, 32, (20, 24)),
])
def test_back_projection_in_the_norm(kind, nx, ny, nz, modes):
    from paper_1111_4971_gb300 import PipeSolver
    a, b = 1.3, 1.0
    if kind == "window":
        geom, hx, hy = Geometry(a, b, 0.13, 0.11, *modes), 0.5 * a / nx, 0.6 * b / ny
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
    source = np.sin(0.47 * np.pi * m)[:, None] * np.sin(0.44 * np.pi * n)[None, :]
    source /= (m[:, None] / a) ** 2 + (n[None, :] / b) ** 2
    source *= (m <= modes[0])[:, None] * (n <= modes[1])[None, :]
    psi = (source[..., None] * (1.0 + 0.3 * np.sin(0.37 * np.arange(nz)))).astype(np.float32)
    phi = s.empty()
    s.stage_modes(2, torch.tensor(psi.reshape(mxp * myp, nz)).cuda(), phi)
    got = phi.double().cpu().numpy()
    want = np.einsum("ny,xnz->xyz", sy, np.einsum("mx,mnz->xnz", sx, psi.astype(np.float64), optimize=True), optimize=True)
    assert np.linalg.norm(got - want) <= 1.25 * 2.0 ** -24 * np.linalg.norm(want)
