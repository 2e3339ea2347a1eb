"""Single stages of the mode-space form touch the caller's buffers only: they run
beside a solve and beside each other on several streams, and in a captured graph."""
import pytest
import torch

from test_gpu_mode_split import make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1111_4971_gb300 import build
    build.build()


def inputs(s, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    part, psi = s.mode_buffers()
    rho = torch.rand(s.shape, dtype=torch.float64, device="cuda", generator=g) - 0.3
    psi = torch.rand(psi.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5
    return rho, psi


def stages(s, rho, psi, stream=None):
    part, _ = s.mode_buffers()
    phi = s.empty()
    s.stage_modes(0, rho, part, stream=stream)
    s.stage_modes(2, psi, phi, stream=stream)
    return part, phi


def test_stages_and_a_solve_on_three_streams():
    s = make("centred", 64, 128, 512, (20, 20))
    data = [inputs(s, k) for k in range(2)]
    want = [stages(s, *d) for d in data]
    want_phi = s.solve(data[0][0])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    got, solved = [[], []], []
    for _ in range(8):
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                got[k].append(stages(s, *data[k]))
        with torch.cuda.stream(streams[2]):
            solved.append(s.solve(data[0][0]))
    torch.cuda.synchronize()
    for k in range(2):
        for part, phi in got[k]:
            assert torch.equal(part, want[k][0]) and torch.equal(phi, want[k][1])
    for phi in solved:
        assert torch.equal(phi, want_phi)


def test_stages_in_a_captured_graph():
    s = make("wall", 32, 48, 64, (7, 9))
    rho, psi = inputs(s, 3)
    want = stages(s, rho, psi)
    torch.cuda.synchronize()
    part, phi = torch.zeros_like(want[0]), torch.zeros_like(want[1])
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(graph, stream=stream):
            s.stage_modes(0, rho, part, stream=stream)
            s.stage_modes(2, psi, phi, stream=stream)
    for _ in range(3):
        part.zero_()
        phi.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(part, want[0]) and torch.equal(phi, want[1])
