"""E = -grad phi in 16-byte pieces: the smallest and ragged meshes, every face,
against numpy.gradient."""
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


# three products and two sums a value, each rounded once: 8 roundings of terms
# of at most 4 max |phi| / 2h
@pytest.mark.parametrize("dtype,u", [(torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)])
@pytest.mark.parametrize("shape", [(16, 16, 32), (16, 48, 64), (80, 16, 1024)])
def test_field_faces_and_pieces(shape, dtype, u):
    from paper_1111_4971_gb300 import PipeSolver
    geom, grid = cell_centred(1.5, 1.0, *shape, 0.03, modes=8)
    s = PipeSolver(geom, grid, dtype=dtype)
    phi = torch.rand(shape, dtype=torch.float64, device="cuda").to(dtype)
    E = s.electric_field(phi).double().cpu().numpy()
    p = phi.double().cpu().numpy()
    for axis, h in enumerate((grid.hx, grid.hy, grid.hz)):
        want = -np.gradient(p, h, axis=axis, edge_order=2)
        assert np.abs(E[axis] - want).max() <= 8 * u * 4 / (2 * h)
