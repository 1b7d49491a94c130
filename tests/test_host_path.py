"""fftn / ifftn without a GPU: which calls skip the autograd Function, and what
happens where torch does not have the internals that decide it."""
import pytest
import torch

from paper_2209_15040_gb300 import wsfft as W


@pytest.fixture
def routes(monkeypatch):
    taken = []
    monkeypatch.setattr(W, "_run", lambda x, *a, **k: taken.append("direct") or x)

    class Function:
        @staticmethod
        def apply(x, *a):
            taken.append("function")
            return x

    monkeypatch.setattr(W, "_FFTN", Function)
    return taken


def test_plain_and_tracked_calls(routes):
    x = torch.zeros(8, dtype=torch.complex64)
    W.fftn(x)
    W.ifftn(x.clone().requires_grad_(True))
    with torch.no_grad():
        W.fftn(x.clone().requires_grad_(True))
    assert routes == ["direct", "function", "direct"]


@pytest.mark.parametrize("missing", ["_functorch_active", "_forward_level"])
def test_without_the_internals_every_call_takes_the_function(routes, monkeypatch, missing):
    monkeypatch.setattr(W, missing, None)
    W.fftn(torch.zeros(8, dtype=torch.complex64))
    assert routes == ["function"]


def test_stream_handle_without_the_raw_getter(monkeypatch):
    class Stream:
        cuda_stream = 1234

    monkeypatch.setattr(W, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    assert W._stream_handle() == 1234
    assert W._stream_handle(77) == 77
