"""The constants that the backward pass of ``cost`` keeps with a handle: their values, made once, and
finished before another call can find them (no GPU: the tensors and the stream are stand-ins)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2007_06427_gb300 import autograd


class Loop:
    L, nx, ns, batch = 22.0, 8, [8, 16, 8], 3


def test_values_made_once():
    loop, cpu = Loop(), torch.device("cpu")
    index = autograd.loop_index(loop, cpu)
    assert index.tolist() == [0] * 64 + [1] * 128 + [2] * 64
    assert autograd.loop_index(loop, cpu) is index
    factor = autograd.loop_factor(loop, cpu)
    assert factor.tolist() == [2 * 22.0 / (8 * n) for n in (8, 16, 8)]
    assert autograd.loop_factor(loop, cpu) is factor


@pytest.mark.parametrize("get", [autograd.loop_index, autograd.loop_factor])
def test_finished_before_it_is_kept(get, monkeypatch):
    loop, kept = Loop(), []

    class Made:
        is_cuda, device = True, "cuda:0"

    class Stream:
        def synchronize(self):
            kept.append(dict(loop.__dict__.get("_cache", {})))

    monkeypatch.setattr(autograd.torch, "tensor", lambda *a, **k: Made())
    monkeypatch.setattr(autograd.torch, "arange", lambda *a, **k: Made())
    monkeypatch.setattr(autograd.torch, "repeat_interleave", lambda *a, **k: Made())
    monkeypatch.setattr(autograd.torch.cuda, "current_stream", lambda device=None: Stream())
    value = get(loop, "cuda:0")
    assert kept == [{}]                      # one wait, with nothing kept yet
    assert get(loop, "cuda:0") is value and len(kept) == 1
