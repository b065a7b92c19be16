"""Host arguments of the binding, without a GPU."""
import ctypes

import pytest
import torch

from paper_2307_14995_b200 import binding as la


def floats(arg, n):
    if isinstance(arg, int):
        return list((ctypes.c_float * n).from_address(arg))
    return list(arg)


@pytest.mark.parametrize("lam", [
    torch.tensor([1.0, 0.5, 0.25]),                            # read where it lies
    torch.tensor([1.0, 9.0, 0.5, 9.0, 0.25, 9.0])[::2],         # a stride
    torch.tensor([1.0, 0.5, 0.25], dtype=torch.float64),
    torch.nn.Parameter(torch.tensor([1.0, 0.5, 0.25])),
    torch._neg_view(torch.tensor([-1.0, -0.5, -0.25])),        # the memory holds the negated values
    [1.0, 0.5, 0.25],
])
def test_decay_rates_reach_the_library_by_value(lam):
    assert floats(la._lam(lam), 3) == [1.0, 0.5, 0.25]


@pytest.mark.parametrize("lam", [torch.tensor(0.5), torch.tensor([[1.0, 0.5]]), torch.ones(2, 1), 0.5])
def test_decay_rates_that_are_no_vector_are_refused(lam):
    with pytest.raises(TypeError):
        la._lam(lam)


@pytest.mark.parametrize("missing", ["_RAW_STREAM", "_CURRENT_DEVICE"])
def test_current_stream_without_the_private_functions(monkeypatch, missing):
    class Stream:
        cuda_stream = 77

    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    monkeypatch.setattr(la, "_RAW_STREAM", lambda device: 5)
    monkeypatch.setattr(la, "_CURRENT_DEVICE", lambda: 0)
    assert la._stream(None) == 5 and la._stream(Stream) == 77
    monkeypatch.setattr(la, missing, None)
    assert la._stream(None) == 77
