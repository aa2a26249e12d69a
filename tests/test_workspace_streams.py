"""A workspace that a call makes for itself belongs to the current stream's pool: when the
call runs on another stream, the allocator has to know of that stream."""
import pytest
import torch

import paper_2004_05962_gb300 as P
from paper_2004_05962_gb300 import bsi as B
from paper_2004_05962_gb300 import synth


class _Tensor:
    is_cuda = True

    def __init__(self, n):
        self.n, self.recorded = n, []

    def numel(self):
        return self.n

    def element_size(self):
        return 1

    def record_stream(self, s):
        self.recorded.append(s)


class _Handle:
    cuda_stream = 7


def test_own_workspace_is_recorded_on_the_given_stream(monkeypatch):
    monkeypatch.setattr(torch, "empty", lambda n, dtype, device: _Tensor(n))
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda ptr, device=None: ("external", ptr, device))
    ws, n = B._workspace(64, "cuda:0", None, _Handle())
    assert n == 64 and ws.recorded == [("external", 7, "cuda:0")]
    assert B._workspace(64, "cuda:0", None, None)[0].recorded == []      # the current stream: nothing to record
    mine = _Tensor(64)
    assert B._workspace(64, "cuda:0", mine, _Handle())[0] is mine and mine.recorded == []   # the caller's, and the caller's to keep
    assert B._workspace(0, "cuda:0", None, _Handle()) == (None, 0)


@pytest.mark.gpu
def test_calls_on_another_stream():
    shape, spacing = (40, 48, 61), (5, 4, 3)
    dev = torch.device("cuda", 0)
    g = torch.from_numpy(synth.normal_field(shape, seed=3)).to(dev)
    phi = torch.from_numpy(synth.uniform_phi(shape, spacing, -2, 2, seed=4)).to(dev)
    image = torch.rand(shape, device=dev)
    side = torch.cuda.Stream()
    calls = [lambda s: P.bsi_field_adjoint(g, spacing, stream=s),
             lambda s: P.bsi_field_adjoint_batched([g, g], [spacing, spacing], stream=s)[1],
             lambda s: P.bsi_field_adjoint_rational(g, (47, 47, 47), (10, 10, 10), stream=s),
             lambda s: P.bsi_resample_backward(phi, shape, spacing, image, g[..., 0].contiguous(), stream=s)]
    for call in calls:
        want = call(None)
        torch.cuda.synchronize()
        for s in (side, torch.cuda.ExternalStream(side.cuda_stream), type("S", (), {"cuda_stream": side.cuda_stream})()):
            side.wait_stream(torch.cuda.current_stream())
            got = call(s)
            torch.cuda.synchronize()
            assert torch.equal(got, want)
