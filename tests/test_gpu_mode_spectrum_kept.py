"""pipe_mode_spectrum computes its table once per handle: later calls are a copy,
from any thread."""
import threading

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


def solver():
    from paper_1111_4971_gb300 import PipeSolver
    return PipeSolver(*cell_centred(1.3, 1.0, 32, 32, 1024, 0.05), igf=True, dtype=torch.float32)


def test_later_calls_are_a_copy():
    """The table stays on the device from the first call until the handle is
    destroyed; later calls allocate nothing."""
    solver().mode_spectrum()                     # (loads the kernels' code)
    s = solver()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    f0 = free()
    table = s.mode_spectrum()
    f1 = free()
    assert f0 - f1 >= table.nbytes
    assert np.array_equal(s.mode_spectrum(), table) and free() == f1
    s.close()
    assert free() >= f0


def test_first_calls_from_several_threads():
    want = solver().mode_spectrum()
    s, got = solver(), []
    threads = [threading.Thread(target=lambda: got.append(s.mode_spectrum())) for _ in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(got) == 6 and all(np.array_equal(g, want) for g in got)
