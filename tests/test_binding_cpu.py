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


def test_argument_kinds_are_those_of_the_header(monkeypatch):
    """Every call on device tensors names its arguments as the C prototype has them."""
    import inspect
    import os
    import re
    header = open(os.path.join(os.path.dirname(la.LIB_PATH), "..", "include", "la.h")).read()
    header = re.sub(r"/\*.*?\*/|//[^\n]*", "", header, flags=re.S)
    want = {}
    for name, args in re.findall(r"la_status\s+(la_\w+)\(([^;]*?)\);", header, re.S):
        kinds = ""
        for a in (" ".join(x.split()) for x in args.split(",")):
            if "la_shape" in a:
                kinds += "s"
            elif a == "void* stream":
                kinds += "r"
            elif a.endswith("_host"):
                kinds += "h"
            else:
                kinds += "t" if "*" in a else "i"
        want[name] = kinds
    want["la_bwd"] = want["la_bwd_reuse"]
    got = []
    monkeypatch.setattr(la, "_enter", lambda name, kinds, *args: got.append((name, kinds, len(args))))
    lam, cu = [1.0], [0, 1]
    for name in ("la_fwd", "la_fwd_gated", "la_gate_fwd", "la_gate_bwd", "la_fwd_noalloc", "la_bwd", "la_decode_step", "la_decode_steps",
                 "la_fwd_varlen", "la_bwd_varlen", "la_chunk_state", "la_chain_states", "la_lrpe_fwd", "la_lrpe_bwd"):
        f = getattr(la, name)
        given = {p: lam if p == "lam" else cu if p == "cu_seqlens" else
                 0 if p in ("reverse", "total_tokens", "chunk_tokens", "num_chunks", "chunk", "pos0") else None
                 for p in inspect.signature(f).parameters}
        f(**given)
        assert got[-1] == (name, want[name], len(want[name]))


@pytest.mark.parametrize("args,error", [
    (("shape", torch.zeros(4)), ValueError),          # a tensor that is not on a GPU
    (("shape", 5), AttributeError),                   # an address instead of a tensor
    (("shape", b"abc"), AttributeError),
    ((5, None), TypeError),                           # an address instead of a shape
    ((None, None), TypeError),
])
def test_arguments_that_are_refused(args, error):
    shape = la.make_shape(1, 1, 1, 64, 64, torch.bfloat16, torch.float32)
    first, q = args
    with pytest.raises(error):
        la.la_decode_step(shape if first == "shape" else first, q, None, None, [1.0], None, None)


def test_first_use_from_several_threads(monkeypatch):
    """No thread may find a call that is ready to be made while the table of addresses still changes."""
    import sys
    import threading
    la.load()
    want = dict(la._address)
    assert want["la_bwd"] == want["la_bwd_reuse"]  # (la_bwd passes the forward pass's workspace too)
    wrong = []

    def first_use(start):
        start.wait()
        if la._call is None:
            la.load()
        for _ in range(50):
            if dict(la._address) != want:
                wrong.append(dict(la._address))

    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        for _ in range(100):
            for name, value in (("_lib", None), ("_call", None), ("_address", {})):
                monkeypatch.setattr(la, name, value)
            start = threading.Barrier(4)
            threads = [threading.Thread(target=first_use, args=(start,)) for _ in range(4)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
    finally:
        sys.setswitchinterval(interval)
    assert not wrong


@pytest.mark.parametrize("handle,want", [(77, 77), (None, 0), (ctypes.c_void_p(77), 77), (ctypes.c_void_p(None), 0)])
def test_streams_of_other_libraries(handle, want):
    """A stream is any object with a handle; what ctypes takes for a pointer is one."""
    class Stream:
        cuda_stream = handle

    got = []
    callback = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p)(lambda p: got.append(p or 0) or 0)
    la.load()
    assert la._call(ctypes.cast(callback, ctypes.c_void_p).value, "r", Stream) == 0
    assert got == [want]


def test_a_stream_that_is_no_handle_is_refused():
    class Stream:
        cuda_stream = 1.5

    la.load()
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        la._call(la._address["la_version"], "r", Stream)


def test_the_extension_module_is_this_interpreters():
    import importlib.machinery
    from paper_2307_14995_b200 import build
    build.build()
    la.load()
    from paper_2307_14995_b200 import _la_call
    suffix = importlib.machinery.EXTENSION_SUFFIXES[0]  # the one with the interpreter's tag
    assert suffix != ".so" and _la_call.__file__.endswith("_la_call" + suffix)
