"""The z stage of the mode-space form (two first-order recurrences per mode
column) against the linear convolution with K_mn(d), element by element.

Sizes: one to four warps a column and the shortest column; kappa*hz from far
below one (long memory, where a rounded q = e^{-kappa hz} would drift) to
large (q underflows in FP32)."""
import numpy as np
import pytest
import torch

from inputs.bunches import Geometry, Grid
from oracle import green

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


# A value passes at most 8 + 8 steps of a recurrence (two roundings each in
# FP32), 5 scan steps, 4 warps and the final sum, on parameters rounded once:
# fewer than 64 roundings, each relative to the sum of |K rho| that it belongs to.
@pytest.mark.parametrize("dtype,u", [(torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)])
@pytest.mark.parametrize("igf", [0, 1])
@pytest.mark.parametrize("nz,hz", [(32, 0.05), (64, 20.0), (256, 1e-5), (512, 0.01), (1024, 1e-4), (1024, 0.02)])
def test_mode_z_recurrence_against_convolution(nz, hz, igf, dtype, u):
    from paper_1111_4971_gb300 import PipeSolver
    geom = Geometry(1.0, 1.3, 0.02, 0.03, 3, 5)
    grid = Grid(32, 16, nz, 0.03, 0.06, hz)
    s = PipeSolver(geom, grid, igf=bool(igf), dtype=dtype)
    s.set_plan(t_kind=3)
    mx, mxp, myp, fold, xb = s.mode_layout()
    rng = np.random.default_rng(nz + igf)
    part, psi = s.mode_buffers()
    part.copy_(torch.tensor(rng.uniform(-1.0, 1.0, part.shape)).to(dtype))
    rho = part.double().cpu().numpy().sum(axis=0).reshape(mxp, myp, nz)
    if fold:
        slots = [2 * q + 1 if q < myp // 2 else 2 * (q - myp // 2) + 2 for q in range(myp)]
    else:
        slots = list(range(1, myp + 1))
    kap = green.kappa(np.arange(1, mxp + 1)[:, None], np.array(slots)[None, :], geom.a, geom.b)
    live = (np.arange(1, mxp + 1)[:, None] <= geom.modes_m) & (np.array(slots)[None, :] <= geom.modes_n)
    d = np.arange(nz) * hz
    K = green.z_profile(d, kap[:, :, None], hz, igf) / kap[:, :, None]
    K = K * green.prefactor_G(geom) * grid.hx * grid.hy * hz * live[:, :, None]
    s.stage_modes(1, part, psi)
    torch.cuda.synchronize()
    got = psi.double().cpu().numpy().reshape(mxp, myp, nz)
    lag = np.abs(np.arange(nz)[:, None] - np.arange(nz)[None, :])
    for m in range(mxp):
        for n in range(myp):
            T = K[m, n][lag]
            scale = np.abs(T) @ np.abs(rho[m, n])
            assert (np.abs(got[m, n] - T @ rho[m, n]) <= 64 * u * scale + 1e-300).all(), (m, n)
