"""States entering the segments of a long sequence against the fp64 oracle.  d = 128: segments that one thread block sums,
that a cluster shares, that the walk chains itself and that reach it as running sums; d = 64: the scan.  And the full-precision
kernels.

Tolerance: on-chip operands are two bf16 terms, 2^-17 of each product; a chain of 57 blocks in one fp32 accumulator adds up
to 912 products with a relative error of 2^-24 of the running sum each.  Against RMS(ref), with |sum| up to 5 RMS: 2^-17 * 5 +
912 * 2^-24 * 5 = 3.1e-4."""
import pytest
import torch

from la_check import assert_close
from oracle import la_oracle as orc
from paper_2307_14995_b200 import binding as la

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,N,seg_len,lam", [
    (1, 8500, 4224, [1.0, 0.9995, 0.9, 1e-30]),   # 33 blocks, unshared; ragged tail
    (1, 4097, 2048, [1.0, 0.9995]),               # shared by a cluster; a tail of one token
    (2, 1211, 128, [1.0, 0.999, 0.5]),            # one block a segment, ten segments: running sums
    (1, 700, 128, [0.9, 1.0, 0.9995]),            # five segments: chained by the walk
    (3, 3001, 0, [1.0, 0.98]),                    # the library's own plan
])
def test_states_entering_segments(B, N, seg_len, lam, d):
    H = len(lam)
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen).bfloat16() for _ in range(4)]
    kv_in, gko = [torch.randn(B, H, d, d, generator=gen) * 0.1 for _ in range(2)]
    lam = torch.tensor(lam)
    dev = [x.cuda() for x in (q, k, v, do, kv_in, gko)]
    o, kv = la.fwd(*dev[:3], lam, out_dtype=torch.float32, kv_in=dev[4], want_state=True, seg_len=seg_len)
    dq, dk, dv, gin = la.bwd(*dev[:4], lam, out_dtype=torch.float32, kv_in=dev[4], grad_kv_out=dev[5], want_state_grad=True,
                             seg_len=seg_len)
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    ref = orc.fwd_rec(q, k, v, lam64, kv_in=kv_in, want_state=True)
    ref += orc.bwd_rec(q, k, v, do, lam64, kv_in=kv_in, grad_kv_out=gko, want_state_grad=True)
    for name, g, r in zip(("o", "kv", "dq", "dk", "dv", "gin"), (o, kv, dq, dk, dv, gin), ref):
        assert_close(g, r, 3.1e-4, name)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N,seg_len,layout", [(1, 0, 0), (33, 0, 1), (256, 0, 0), (257, 0, 1), (700, 512, 0), (641, 640, 0)])
def test_full_precision_rows(d, N, seg_len, layout):
    """fp32 inputs: row tiles by themselves (segments up to 512 tokens) and the block-by-block walk (640).  Sums of at most
    640 + d fp32 products each: 768 * 2^-24 of the largest partial sum, itself at most 2 RMS: 9.2e-5."""
    H = 3
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(2, H, N, d, generator=gen) * d ** -0.5 for _ in range(4)]
    kv_in, gko = [torch.randn(2, H, d, d, generator=gen) * 0.1 for _ in range(2)]
    lam = torch.tensor([1.0, 0.97, 1e-20])
    lam64 = lam.double().numpy()
    ref = orc.fwd_rec(q, k, v, lam64, kv_in=kv_in, want_state=True)
    ref += orc.bwd_rec(q, k, v, do, lam64, kv_in=kv_in, grad_kv_out=gko, want_state_grad=True)
    dev = [x.cuda() for x in (q, k, v, do)]
    if layout:
        dev = [x.transpose(1, 2).contiguous() for x in dev]
    shape = la.make_shape(2, H, N, d, d, torch.float32, torch.float32, seg_len, la.LA_PATH_SIMT,
                          layout=la.LA_LAYOUT_BNHD if layout else la.LA_LAYOUT_BHND)
    o, dq, dk, dv = [torch.empty_like(x) for x in dev]
    kv, gin = [torch.empty(2, H, d, d, device="cuda") for _ in range(2)]
    la.la_fwd(shape, *dev[:3], lam, o, kv_in.cuda(), kv, la.alloc_workspace(la.LA_OP_FWD, shape, "cuda"))
    la.la_bwd(shape, *dev, lam, dq, dk, dv, kv_in.cuda(), gko.cuda(), gin, la.alloc_workspace(la.LA_OP_BWD, shape, "cuda"))
    torch.cuda.synchronize()
    back = (lambda x: x.transpose(1, 2)) if layout else (lambda x: x)
    for name, g, r in zip(("o", "kv", "dq", "dk", "dv", "gin"), (back(o), kv, back(dq), back(dk), back(dv), gin), ref):
        assert_close(g, r, 9.2e-5, name)


@pytest.mark.parametrize("d,T,layout", [(64, 8, 0), (128, 8, 1), (64, 9, 1), (128, 17, 0)])
def test_decode_token_counts(d, T, layout):
    """One chunk of tokens on chip, one more than that, two and one more.  Each o adds d fp32 products of a state that has
    been rounded at most T times: (d + 2 T) * 2^-24 of up to 8 RMS, at most 7.8e-5."""
    B, H = 2, 3
    gen = torch.Generator().manual_seed(T)
    q, k, v = [torch.randn(B, H, T, d, generator=gen).bfloat16() for _ in range(3)]
    kv0 = torch.randn(B, H, d, d, generator=gen)
    lam = torch.tensor([1.0, 0.97, 1e-20])
    state = kv0.double().numpy().copy()
    ref = [orc.decode_step(q[:, :, t], k[:, :, t], v[:, :, t], lam.double().numpy(), state) for t in range(T)]
    move = (lambda x: x.transpose(1, 2).contiguous()) if layout else (lambda x: x)
    shape = la.make_shape(B, H, T, d, d, torch.bfloat16, torch.float32, layout=la.LA_LAYOUT_BNHD if layout else la.LA_LAYOUT_BHND)
    dev = [move(x).cuda() for x in (q, k, v)]
    kv, o = kv0.cuda(), torch.empty(dev[0].shape, device="cuda")
    la.la_decode_steps(shape, *dev, lam, kv, o)
    for t in range(T):
        assert_close(move(o)[:, :, t:t + 1], ref[t][:, :, None, :], 7.8e-5, "o[%d]" % t)
    assert_close(kv, state, 7.8e-5, "state")


@pytest.mark.parametrize("d,B,N,seg_len,lam", [
    (128, 1, 4300, 0, [1.0, 0.9995, 0.97, 1e-30]),      # the library's own plan: segments shared by clusters, a ragged tail
    (128, 2, 777, 0, [1.0] * 16),                       # one segment of seven blocks, whose last is short
    (128, 1, 8500, 4224, [1.0, 0.9995, 0.999, 0.9]),    # 33 blocks: shared by two at most
    (128, 1, 1211, 128, [1.0, 0.999, 0.5]),             # ten pieces in the chain, the last one shorter
    (128, 1, 5, 0, [1.0, 0.5]),
    (64, 1, 1211, 128, [1.0, 0.999, 0.5]),
])
def test_chunk_state(d, B, N, seg_len, lam):
    H = len(lam)
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen).bfloat16() for _ in range(4)]
    lam = torch.tensor(lam)
    shape = la.make_shape(B, H, N, d, d, torch.bfloat16, torch.float32, seg_len)
    ws = torch.empty(la.chunk_state_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    kv, gin = [torch.empty(B, H, d, d, device="cuda") for _ in range(2)]
    la.la_chunk_state(shape, 0, k.cuda(), v.cuda(), lam, kv, ws)
    la.la_chunk_state(shape, 1, q.cuda(), do.cuda(), lam, gin, ws)
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    assert_close(kv, orc.fwd_rec(q, k, v, lam64, want_state=True)[1], 3.1e-4, "forward")
    assert_close(gin, orc.bwd_rec(q, k, v, do, lam64, want_state_grad=True)[3], 3.1e-4, "reverse")


@pytest.mark.parametrize("d,B,H,N", [(64, 8, 24, 640), (64, 1, 4, 512), (64, 1, 2, 513), (128, 5, 16, 333), (128, 1, 2, 1300), (128, 40, 8, 1100)])
def test_full_precision_plans(d, B, H, N):
    """The library's own segments for fp32 inputs: few heads and many, one segment of row tiles, several, the walk.  Sums of
    at most N + d fp32 products: 1428 * 2^-24 of the largest partial sum, itself at most 2 RMS: 1.7e-4."""
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen) * d ** -0.5 for _ in range(4)]
    lam = torch.linspace(0.6, 1.0, H)
    dev = [x.cuda() for x in (q, k, v, do)]
    o = la.fwd(*dev[:3], lam)
    grads = la.bwd(*dev, lam)
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    ref = (orc.fwd_rec(q, k, v, lam64),) + tuple(orc.bwd_rec(q, k, v, do, lam64))
    for name, g, r in zip(("o", "dq", "dk", "dv"), (o,) + tuple(grads), ref):
        assert_close(g, r, 1.7e-4, name)


@pytest.mark.parametrize("d,dtype,sets", [(128, torch.bfloat16, (1, 2)), (64, torch.bfloat16, (2, 3)), (128, torch.float32, (2, 3))])
@pytest.mark.parametrize("B,N,seg_len", [(1, 1211, 128), (2, 700, 256)])
def test_workspace_holds_the_sets_that_are_used(d, dtype, sets, B, N, seg_len):
    """Nothing behind la_workspace_bytes is written, a byte less is refused, and the backward pass from the forward pass's
    states (with more than six segments at d = 128: running sums, read transposed) agrees with the oracle."""
    lam = torch.tensor([1.0, 0.999, 0.5])
    H = len(lam)
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen).to(dtype) for _ in range(4)]
    kv_in, gko = [torch.randn(B, H, d, d, generator=gen) * 0.1 for _ in range(2)]
    shape = la.make_shape(B, H, N, d, d, dtype, torch.float32, seg_len)
    state = B * H * d * d * 4 * -(-N // seg_len)
    need = [la.workspace_bytes(op, shape) for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    assert need == [n * state for n in sets]
    bufs = [torch.full((n + 4096,), 0xA5, dtype=torch.uint8, device="cuda") for n in need]
    ws_f, ws_b = bufs[0][:need[0]], bufs[1][:need[1]]
    dev = [x.cuda() for x in (q, k, v, do, kv_in, gko)]
    o, dq, dk, dv = [torch.empty(B, H, N, d, device="cuda") for _ in range(4)]
    kv, gin = [torch.empty(B, H, d, d, device="cuda") for _ in range(2)]
    with pytest.raises(la.LaError):
        la.la_fwd(shape, *dev[:3], lam, o, dev[4], kv, ws_f[:-1])
    with pytest.raises(la.LaError):
        la.la_bwd(shape, *dev[:4], lam, dq, dk, dv, dev[4], dev[5], gin, ws_b[:-1])
    la.la_fwd(shape, *dev[:3], lam, o, dev[4], kv, ws_f)
    lam64 = lam.double().numpy()
    ref = orc.bwd_rec(q, k, v, do, lam64, kv_in=kv_in, grad_kv_out=gko, want_state_grad=True)
    for reuse in (ws_f, None):
        la.la_bwd(shape, *dev[:4], lam, dq, dk, dv, dev[4], dev[5], gin, ws_b, fwd_workspace=reuse)
        for name, g, r in zip(("dq", "dk", "dv", "gin"), (dq, dk, dv, gin), ref):
            assert_close(g, r, 3.1e-4, name)
    assert all(bool((b[n:] == 0xA5).all()) for b, n in zip(bufs, need))


@pytest.mark.parametrize("lens", [[2600, 700, 1025, 3], [1, 1024, 2048, 2049, 5000]])
def test_packed_segments_shared_by_clusters(lens):
    """Packed sequences in segments of eight blocks, which clusters share, with clusters whose segment a shorter sequence does
    not have, sequences taken longest first, and a tail of one and of three tokens."""
    H, d, S = 3, 128, len(lens)
    cu = [sum(lens[:i]) for i in range(S + 1)]
    T = cu[-1]
    gen = torch.Generator().manual_seed(T)
    q, k, v, do = [torch.randn(1, T, H, d, generator=gen).bfloat16() for _ in range(4)]
    kv_in, gko = [torch.randn(S, H, d, d, generator=gen) * 0.1 for _ in range(2)]
    lam = torch.tensor([1.0, 0.9995, 0.9])
    shape = la.make_shape(1, H, T, d, d, torch.bfloat16, torch.float32, 1024, layout=la.LA_LAYOUT_BNHD)
    dev = [x.cuda() for x in (q, k, v, do, kv_in, gko)]
    o, dq, dk, dv = [torch.empty(1, T, H, d, device="cuda") for _ in range(4)]
    kv, gin = [torch.empty(S, H, d, d, device="cuda") for _ in range(2)]
    ws = [torch.empty(la.varlen_workspace_bytes(op, shape, cu), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    la.la_fwd_varlen(shape, *dev[:3], lam, o, cu, dev[4], kv, ws[0])
    la.la_bwd_varlen(shape, *dev[:4], lam, dq, dk, dv, cu, dev[4], dev[5], gin, ws[1])
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    for i in range(S):
        part = lambda x: x[:, cu[i]:cu[i + 1]].transpose(1, 2)
        one = [part(x).contiguous() for x in (q, k, v, do)]
        ref = orc.fwd_rec(*one[:3], lam64, kv_in=kv_in[i:i + 1], want_state=True)
        ref += orc.bwd_rec(*one, lam64, kv_in=kv_in[i:i + 1], grad_kv_out=gko[i:i + 1], want_state_grad=True)
        got = (part(o), kv[i:i + 1], part(dq), part(dk), part(dv), gin[i:i + 1])
        for name, g, r in zip(("o", "kv", "dq", "dk", "dv", "gin"), got, ref):
            assert_close(g, r, 3.1e-4, "%s of sequence %d" % (name, i))


@pytest.mark.parametrize("B,H,N,d", [(8, 16, 200, 64), (8, 8, 200, 128), (1, 1, 31, 64), (1, 1, 480, 128), (1, 5, 1100, 64)])
def test_full_precision_tiles_shared_by_groups_or_not(B, H, N, d):
    """Few thread blocks share their tiles out over groups of threads, many do not.  Sums of at most N + d products: (N + d) *
    2^-24 of the largest partial sum, at most 5 RMS: 3.6e-4."""
    gen = torch.Generator().manual_seed(N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen) * d ** -0.5 for _ in range(4)]
    lam = torch.linspace(0.3, 1.0, H)
    dev = [x.cuda() for x in (q, k, v, do)]
    o, kv = la.fwd(*dev[:3], lam, want_state=True)
    grads = la.bwd(*dev, lam)
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    ref = tuple(orc.fwd_rec(q, k, v, lam64, want_state=True)) + tuple(orc.bwd_rec(q, k, v, do, lam64))
    for name, g, r in zip(("o", "kv", "dq", "dk", "dv"), (o, kv) + tuple(grads), ref):
        assert_close(g, r, 3.6e-4, name)


@pytest.mark.parametrize("B,H,N,d", [
    (1, 25, 400, 128), (1, 8, 300, 128), (2, 32, 512, 128), (1, 75, 512, 128), (4, 25, 128, 128), (5, 30, 64, 128),  # one group or two,
    (5, 28, 128, 128), (1, 90, 300, 128), (1, 55, 512, 128), (2, 50, 160, 128),                                      # two at a time
    (1, 45, 512, 64), (1, 19, 500, 64), (1, 90, 300, 64), (1, 70, 300, 64), (5, 28, 128, 64), (4, 50, 64, 64)])      # one or four
def test_full_precision_groups_by_the_tiles_of_a_row(B, H, N, d):
    """On both sides of where a launch's tiles are shared out, by how many a row adds up.  Tolerance as above: at most 640 products."""
    gen = torch.Generator().manual_seed(B * H * N)
    q, k, v, do = [torch.randn(B, H, N, d, generator=gen) * d ** -0.5 for _ in range(4)]
    lam = torch.linspace(0.5, 1.0, H)
    dev = [x.cuda() for x in (q, k, v, do)]
    o = la.fwd(*dev[:3], lam)
    grads = la.bwd(*dev, lam)
    torch.cuda.synchronize()
    lam64 = lam.double().numpy()
    ref = (orc.fwd_rec(q, k, v, lam64),) + tuple(orc.bwd_rec(q, k, v, do, lam64))
    for name, g, r in zip(("o", "dq", "dk", "dv"), (o,) + tuple(grads), ref):
        assert_close(g, r, 3.6e-4, name)
