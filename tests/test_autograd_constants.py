"""The constants that the backward pass of ``cost`` keeps with a handle (no GPU: the streams are
stand-ins): their values, once per stream, since those that one stream made need not be complete on
another, and under capture the ones that are there."""
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import autograd

CPU = torch.device("cpu")


class Loop:
    L, nx, ns, batch = 22.0, 8, [8, 16, 8], 3


class Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


def test_values():
    factor, index = autograd.constants(Loop(), CPU, Stream(1))
    assert index.tolist() == [0] * 64 + [1] * 128 + [2] * 64
    assert factor.tolist() == [2 * 22.0 / (8 * n) for n in (8, 16, 8)]


def test_once_per_stream(monkeypatch):
    monkeypatch.setattr(autograd.torch.cuda, "is_current_stream_capturing", lambda: False)
    loop = Loop()
    a = autograd.constants(loop, CPU, Stream(1))
    b = autograd.constants(loop, CPU, Stream(2))
    assert a[1] is not b[1] and torch.equal(a[1], b[1])
    assert autograd.constants(loop, CPU, Stream(1)) is a and autograd.constants(loop, CPU, Stream(2)) is b


def test_capture_takes_what_is_there(monkeypatch):
    loop = Loop()
    a = autograd.constants(loop, CPU, Stream(1))
    monkeypatch.setattr(autograd.torch.cuda, "is_current_stream_capturing", lambda: True)
    assert autograd.constants(loop, CPU, Stream(2)) is a
    monkeypatch.setattr(autograd.torch.cuda, "is_current_stream_capturing", lambda: False)
    assert autograd.constants(loop, CPU, Stream(2)) is not a
