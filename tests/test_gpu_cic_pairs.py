"""FP32 deposit by 4-wide reductions: every position of a pair of z nodes within
16 bytes, both ends of the mesh in z and outside it, and a field that is only
4-byte aligned, against a 64-bit deposit."""
import ctypes

import numpy as np
import pytest
import torch

from inputs.bunches import cell_centred

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


@pytest.mark.parametrize("offset", [0, 1])       # floats past a 16-byte boundary
def test_deposit_pairs(offset):
    from paper_1111_4971_gb300 import PipeSolver
    geom, grid = cell_centred(1.0, 1.0, 16, 16, 32, 0.25)
    s = PipeSolver(geom, grid, dtype=torch.float32)
    rng = np.random.default_rng(3)
    n, q = 1500, 0.5
    # z/hz in eighths, so that cells and weights are exact; -1.5 .. 33 covers both ends
    k = rng.integers(-12, 8 * 33, n) / 8.0
    xyz = np.stack([rng.integers(-8, 136, n) / 128.0, rng.integers(-8, 136, n) / 128.0, k * grid.hz], 1)
    x = torch.tensor(xyz, dtype=torch.float32, device="cuda")
    buf = torch.full((grid.nx * grid.ny * grid.nz + 8,), 0.25, device="cuda")
    field = buf[offset:offset + grid.nx * grid.ny * grid.nz]
    assert s.lib.pipe_cic_deposit(s.handle, ctypes.c_void_p(x.data_ptr()), n, q, ctypes.c_void_p(field.data_ptr()),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    want = np.full(grid.shape, 0.25)
    f = np.stack([(xyz[:, 0] - geom.x0) / grid.hx, (xyz[:, 1] - geom.y0) / grid.hy, xyz[:, 2] / grid.hz], 1)
    i0 = np.floor(f).astype(int)
    d = f - i0
    mass = np.zeros(grid.shape)
    for c in range(8):
        o = np.array([c >> 2 & 1, c >> 1 & 1, c & 1])
        w = np.where(o == 1, d, 1 - d).prod(1) * q / (grid.hx * grid.hy * grid.hz)
        i = i0 + o
        ok = ((i >= 0) & (i < np.array(grid.shape))).all(1)
        np.add.at(want, tuple(i[ok].T), w[ok])
        np.add.at(mass, tuple(i[ok].T), np.abs(w[ok]))
    got = field.double().cpu().numpy().reshape(grid.shape)
    # weights and their products: 8 roundings a term; sums: one rounding a term of
    # at most the node's total, fewer than 64 terms a node
    assert (np.abs(got - want) <= 72 * 2.0 ** -24 * (mass + 0.25)).all()
    rest = torch.cat([buf[:offset], buf[offset + field.numel():]])
    assert (rest == 0.25).all()
