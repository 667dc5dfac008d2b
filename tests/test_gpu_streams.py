"""Calls without a stream argument run on torch's current stream: its handle,
and a call captured with the work around it."""
import numpy as np
import pytest
import torch

from paper_2202_08778_gb300 import vet

pytestmark = pytest.mark.gpu


def test_current_stream_is_taken():
    torch.zeros(1, device="cuda")
    assert (vet._stream(None) or 0) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert vet._stream(None) == side.cuda_stream
        assert vet._stream(7) == 7


def test_capture_takes_the_call():
    n = 8
    kappa, E = torch.rand(n, n, n, device="cuda"), torch.zeros(n ** 3, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        doubled = kappa * 2
        vet.point_source((n, n, n), 0.5, (1.0, 1.1, 1.2), 1.0, doubled, E)
        out = E + 1
    assert not E.any()
    graph.replay()
    want = torch.zeros_like(E)
    vet.point_source((n, n, n), 0.5, (1.0, 1.1, 1.2), 1.0, kappa * 2, want)
    torch.cuda.synchronize()
    assert want.all() and torch.equal(out, want + 1)
    with pytest.raises(TypeError):
        vet.point_source((n, n, n), 0.5, (1.0, 1.1, 1.2), 1.0, kappa.double(), E)
    with pytest.raises(TypeError):
        vet.point_source((n, n, n), 0.5, (1.0, 1.1, 1.2), 1.0, np.zeros((n, n, n)), E)
