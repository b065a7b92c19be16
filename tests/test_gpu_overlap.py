"""Launches that begin while the ones before them on the stream end: whatever is read must be complete by then.  Each call reads
what the one before it wrote, nothing waits in between, and the results are those of the same calls with a device-wide wait after
each; likewise when the sequence is replayed from a CUDA graph."""
import pytest
import torch

from paper_2307_14995_b200 import binding as la, inputs

pytestmark = pytest.mark.gpu


def buffers(B, H, N, d, seed, dtype=torch.bfloat16):
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    new = lambda t: (torch.randn(B, H, N, d, generator=gen, device="cuda") * d ** -0.5).to(t)
    shape = la.make_shape(B, H, N, d, d, dtype, dtype)
    x = [new(dtype) for _ in range(9)]  # q k v | o do | dq dk dv | second o
    ws = [torch.empty(max(256, la.workspace_bytes(op, shape)), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    kv = [torch.zeros(B, H, d, d, device="cuda") for _ in range(2)]
    return shape, x, ws, kv


def sequence(shape, x, ws, kv, lam, wait):
    q, k, v, o, do, dq, dk, dv, o2 = x
    reuse = dict(fwd_workspace=ws[0]) if la.workspace_bytes(la.LA_OP_FWD, shape) else {}
    steps = [
        lambda: la.la_fwd(shape, q, k, v, lam, o, None, kv[0], ws[0]),
        lambda: la.la_gate_bwd(shape, o, v, q, do, o2),                                # from o
        lambda: la.la_bwd(shape, q, k, v, do, lam, dq, dk, dv, workspace=ws[1], **reuse),  # from do and the forward states
        lambda: la.la_fwd(shape, dq, dk, dv, lam, o2, kv[0], kv[1], ws[0]),              # from all gradients and the state
        lambda: la.la_bwd(shape, dq, dk, dv, o2, lam, q, k, v, kv_in=kv[0], workspace=ws[1]),
        lambda: la.la_fwd(shape, q, k, v, lam, o, kv[1], kv[0], ws[0]),
    ]
    for f in steps:
        f()
        if wait:
            torch.cuda.synchronize()


@pytest.mark.parametrize("B,H,N,d,dtype", [
    (1, 8, 2048, 128, torch.bfloat16), (2, 4, 300, 128, torch.bfloat16), (1, 16, 1100, 64, torch.bfloat16), (1, 2, 100, 64, torch.bfloat16),
    (1, 4, 600, 64, torch.float32)])
def test_calls_that_read_one_another(B, H, N, d, dtype):
    lam = inputs.decay_rates(H, 0.5)
    want = None
    for wait in (True, False, False, False):
        shape, x, ws, kv = buffers(B, H, N, d, 3, dtype)
        torch.cuda.synchronize()
        sequence(shape, x, ws, kv, lam, wait)
        torch.cuda.synchronize()
        got = [t.clone() for t in x + kv]
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    la.device_status()
    shape, x, ws, kv = buffers(B, H, N, d, 3, dtype)
    start = [t.clone() for t in x + kv]
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        sequence(shape, x, ws, kv, lam, False)
    for _ in range(2):
        for t, s in zip(x + kv, start):
            t.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, x + kv))
    la.device_status()
