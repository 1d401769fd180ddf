"""The binding hands the library the stream that is current where the call is made."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_calls_run_on_the_current_stream(lib):
    side = torch.cuda.Stream()
    assert lib._stream() == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert lib._stream() == side.cuda_stream
    assert lib._stream(side) == side.cuda_stream
    # captured on the side stream: a launch on any other one would end the capture with an error
    phi, psi = torch.rand(2, 17 * 9, dtype=torch.float64, device="cuda").unbind(0)
    want = lib.morphology_project(phi, psi, 16, 8, 1.0, 1.0, 20, 10)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        got = lib.morphology_project(phi, psi, 16, 8, 1.0, 1.0, 20, 10)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
