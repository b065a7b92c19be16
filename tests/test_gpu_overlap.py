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


def everything(d, wait):
    """Every kind of call that launches early, each from what the ones before it wrote, on one workspace per pass; and in between
    launches that do not begin early (more thread blocks than multiprocessors)."""
    H, T, dtype = 16, 1300, torch.bfloat16
    gen = torch.Generator("cuda")
    gen.manual_seed(d)
    new = lambda: (torch.randn(1, T, H, d, generator=gen, device="cuda") * d ** -0.5).to(dtype)
    q, k, v, u, o, o2, y, d_o, du, dq, dk, dv = x = [new() for _ in range(12)]
    kv = [torch.zeros(1, H, d, d, device="cuda") for _ in range(3)]
    kvs, part, dtheta = torch.zeros(3, H, d, d, device="cuda"), torch.zeros(1, H, d, d, device="cuda"), torch.zeros(H, d, device="cuda")
    theta = inputs.make_theta(H, d, seed=1).cuda()
    lam, cu = inputs.decay_rates(H, 0.5), [0, 500, 501, T]
    shape = la.make_shape(1, H, T, d, d, dtype, dtype, layout=la.LA_LAYOUT_BNHD)
    plain = la.make_shape(1, H, T, d, d, dtype, dtype, 128, layout=la.LA_LAYOUT_BNHD)  # 176 thread blocks
    step = la.make_shape(1, H, 1, d, d, dtype, dtype)
    need = [max(la.workspace_bytes(op, shape), la.workspace_bytes(op, plain), la.varlen_workspace_bytes(op, shape, cu),
                la.lrpe_workspace_bytes(op, shape), la.chunk_state_workspace_bytes(shape)) for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    wf, wb = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in need]
    norm = lambda *t: [lambda t=t: la.la_gate_fwd(shape, t, u, t) for t in t]  # in place: the numbers stay in range
    calls = [
        lambda: la.la_fwd_varlen(shape, q, k, v, lam, o, cu, None, kvs, wf),
        lambda: la.la_fwd_gated(shape, o, k, v, u, lam, y, o2, kv_out=kv[0], workspace=wf),
        lambda: la.la_gate_bwd(shape, o2, u, y, d_o, du), *norm(o2, d_o),
        lambda: la.la_bwd_varlen(shape, o2, k, v, d_o, lam, dq, dk, dv, cu, workspace=wb), *norm(dq, dk, dv),
        lambda: la.la_lrpe_fwd(shape, dq, dk, dv, theta, lam, o, workspace=wf), *norm(o),
        lambda: la.la_fwd(plain, o, dk, dv, lam, y, kv[0], kv[1], wf), *norm(y),
        lambda: la.la_lrpe_bwd(shape, o, k, y, d_o, theta, lam, dq, dk, dv, dtheta, workspace=wb), *norm(dq, dk),
        lambda: la.la_bwd(plain, dq, dk, v, o, lam, o2, q, k, workspace=wb), *norm(q, k),
        lambda: la.la_chunk_state(shape, 0, k, v, lam, part, wf),
        lambda: la.la_chain_states(shape, 3 * T, T, 0, kvs, 3, 2, part, lam, kv[2]),
        lambda: la.la_fwd_gated(plain, q, k, v, u, lam, y, kv_in=kv[2], kv_out=kv[0], workspace=wf),
        lambda: la.la_gate_fwd(shape, o, y, d_o),
    ] + [lambda t=t: la.la_decode_step(step, y[:, t], d_o[:, t], v[:, t], lam, kv[0], o[:, t]) for t in range(6)] + [
        lambda: la.la_fwd(shape, o, d_o, v, lam, du, kv[0], kv[1], wf),
    ]
    tensors = x + kv + [kvs, part, dtheta]

    def run():
        for f in calls:
            f()
            if wait:
                torch.cuda.synchronize()

    return run, tensors


@pytest.mark.parametrize("d", [64, 128])
def test_every_kind_of_call_in_one_stream(d):
    want = None
    for wait in (True, False, False, False):
        run, tensors = everything(d, wait)
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        want = want or [t.clone() for t in tensors]
        assert all(bool(t.float().abs().amax() < 1e20) for t in tensors)  # (no NaN, which equals nothing, either)
        assert all(torch.equal(a, b) for a, b in zip(want, tensors))
    la.device_status()
    run, tensors = everything(d, False)
    start = [t.clone() for t in tensors]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        run()
    for _ in range(2):
        for t, s in zip(tensors, start):
            t.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, tensors))
    la.device_status()
