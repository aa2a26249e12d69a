"""Which stream a call takes when none is given, on the CPU: every form of a device
that torch.cuda.current_stream takes, with and without torch's raw-handle call."""
import pytest
import torch

from paper_2004_05962_gb300 import bsi as B


class _Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


@pytest.fixture
def current(monkeypatch):
    """Devices torch.cuda.current_stream was asked for (it answers with handle 5)."""
    asked = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: (asked.append(device), _Stream(5))[1])
    return asked


@pytest.mark.parametrize("device", [None, 0, 1, "cuda", "cuda:1", torch.device("cuda"), torch.device("cpu", 0)], ids=str)
def test_other_forms_of_a_device_ask_torch(current, device):
    assert B._stream(None, device) == 5
    assert current == [device]


def test_a_tensors_device_takes_the_raw_handle(current, monkeypatch):
    monkeypatch.setattr(B, "_raw_stream", lambda index: 40 + index, raising=False)
    assert B._stream(None, torch.device("cuda", 2)) == 42 and current == []


def test_without_the_raw_handle_call(current, monkeypatch):
    monkeypatch.setattr(B, "_raw_stream", None, raising=False)
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert B._stream(None, torch.device("cuda", 1)) == 5 and current == [torch.device("cuda", 1)]


def test_a_given_stream_is_taken(current):
    assert B._stream(_Stream(7), torch.device("cuda", 0)) == 7 and current == []


@pytest.mark.parametrize("raw", [lambda index: 40 + index, None], ids=["raw", "no_raw"])
def test_entry_points_take_the_tensors_stream(current, monkeypatch, raw):
    monkeypatch.setattr(B, "_raw_stream", raw)
    assert B._tensor_stream(None, torch.device("cuda", 2)) == (42 if raw else 5)
    assert B._tensor_stream(_Stream(7), torch.device("cuda", 2)) == 7
