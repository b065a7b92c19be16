"""d = 64 on the tensor cores: packed batches in one set of launches, and what the walk does at the ends of sequences.

Tolerance as for the segment states: two-term operands, 2^-17 of each product, sums of up to 8 blocks; against RMS(ref) with
|sum| up to 5 RMS 1.7e-4.  bf16 results: 2^-8 |ref| besides."""
import numpy as np
import pytest
import torch

from oracle import la_oracle as orc
from paper_2307_14995_b200 import binding as la

pytestmark = pytest.mark.gpu
H, D, LAM = 3, 64, torch.tensor([1.0, 0.97, 0.2])


def packed(lens, dtype, seg_len, seed, states=False):
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    gen = torch.Generator().manual_seed(seed)
    x = [torch.randn(1, cu[-1], H, D, generator=gen).bfloat16() for _ in range(4)]
    extra = [torch.randn(len(lens), H, D, D, generator=gen) * 0.1 for _ in range(2)] if states else [None, None]
    return cu, x, extra, la.make_shape(1, H, cu[-1], D, D, torch.bfloat16, dtype, seg_len, layout=la.LA_LAYOUT_BNHD)


def run(cu, x, extra, shape, dtype, workspace=True):
    q, k, v, do = [t.cuda() for t in x]
    kv_in, gko = [None if t is None else t.cuda() for t in extra]
    S = len(cu) - 1
    o, dq, dk, dv = [torch.full_like(q, float("nan"), dtype=dtype) for _ in range(4)]
    kv, gin = [torch.empty(S, H, D, D, device="cuda") for _ in range(2)]
    ws = [torch.empty(la.varlen_workspace_bytes(op, shape, cu), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    n = la.launch_count()
    la.la_fwd_varlen(shape, q, k, v, LAM, o, cu, kv_in, kv, ws[0] if workspace else None)
    n = la.launch_count() - n
    la.la_bwd_varlen(shape, q, k, v, do, LAM, dq, dk, dv, cu, kv_in, gko, gin, ws[1])
    torch.cuda.synchronize()
    la.device_status()
    return [t.cpu() for t in (o, dq, dk, dv, kv, gin)], n


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("seg_len,states", [(0, False), (256, True), (128, False)])
def test_packed_sequences(dtype, seg_len, states):
    lens = [300, 1, 127, 128, 129, 1000, 64, 513]
    cu, x, extra, shape = packed(lens, dtype, seg_len, 5, states)
    got, launches = run(cu, x, extra, shape, dtype)
    assert launches == (3 if seg_len else 1)
    lam64 = LAM.double().numpy()
    heads = lambda t: t.permute(0, 2, 1, 3)
    for i in range(len(lens)):
        at = slice(cu[i], cu[i + 1])
        q, k, v, do = [heads(t[:, at]) for t in x]
        kv_in, gko = [None if t is None else t[i:i + 1] for t in extra]
        ref = dict(zip(("o", "kv"), orc.fwd_rec(q, k, v, lam64, kv_in=kv_in, want_state=True)))
        ref.update(zip(("dq", "dk", "dv", "gin"), orc.bwd_rec(q, k, v, do, lam64, kv_in=kv_in, grad_kv_out=gko, want_state_grad=True)))
        for name, t in zip(("o", "dq", "dk", "dv", "kv", "gin"), got):
            g = (t[i:i + 1] if name in ("kv", "gin") else heads(t[:, at])).double().numpy()
            r = ref[name]
            rms = np.sqrt(np.mean(r * r, axis=(2, 3), keepdims=True))
            slack = 2.0 ** -8 * np.abs(r) if dtype == torch.bfloat16 and name not in ("kv", "gin") else 0.0
            assert np.all(np.abs(g - r) <= 1.7e-4 * rms + slack), (name, i)


@pytest.mark.parametrize("seg_len", [0, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_packed_sequence_does_not_see_its_neighbours(bad, seg_len):
    cu, x, extra, shape = packed([200, 77, 300], torch.float32, seg_len, 6)
    clean, _ = run(cu, x, extra, shape, torch.float32)
    for t in x:
        t[:, cu[1]:cu[2]] = bad
    dirty, _ = run(cu, x, extra, shape, torch.float32)
    for name, a, b in zip(("o", "dq", "dk", "dv", "kv", "gin"), clean, dirty):
        for i in (0, 2):
            at = (slice(i, i + 1),) if name in ("kv", "gin") else (slice(None), slice(cu[i], cu[i + 1]))
            assert torch.equal(a[at], b[at]), (name, i)


def test_packed_sequences_without_a_workspace_run_one_by_one():
    cu, x, extra, shape = packed([100, 60, 128], torch.float32, 0, 7)
    with_ws, one = run(cu, x, extra, shape, torch.float32)
    without, each = run(cu, x, extra, shape, torch.float32, workspace=False)
    assert (one, each) == (1, 3) and torch.equal(with_ws[0], without[0]) and torch.equal(with_ws[4], without[4])


@pytest.mark.parametrize("precision", [0, 1, 2, 4, 7])
@pytest.mark.parametrize("N", [1, 128, 129, 500])
def test_state_after_the_last_block(N, precision):
    """The two halves that the state is kept in, with and without lo terms: single terms round to 2^-9 of each product."""
    gen = torch.Generator().manual_seed(N)
    q, k, v = [torch.randn(2, H, N, D, generator=gen).bfloat16() for _ in range(3)]
    o, kv = la.fwd(q.cuda(), k.cuda(), v.cuda(), LAM, want_state=True, precision=precision)
    torch.cuda.synchronize()
    ref = orc.fwd_rec(q, k, v, LAM.double().numpy(), want_state=True)
    tol = 1.7e-4 if precision == 7 else 5 * 2.0 ** -8
    for g, r in zip((o, kv), ref):
        rms = np.sqrt(np.mean(r * r, axis=(2, 3), keepdims=True))
        assert np.all(np.abs(g.cpu().double().numpy() - r) <= tol * rms + 2 * tol * np.abs(r))


@pytest.mark.parametrize("d", [64, 128])
def test_packed_calls_in_a_graph(d):
    """A captured call keeps its own copy of the sequences' places."""
    lens = [300, 1, 127, 128, 700, 5]
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    T = cu[-1]
    shape = la.make_shape(1, H, T, d, d, torch.bfloat16, torch.float32, 256, layout=la.LA_LAYOUT_BNHD)
    ws = [torch.empty(la.varlen_workspace_bytes(op, shape, cu), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    gen = torch.Generator().manual_seed(9)
    inputs = [[torch.randn(1, T, H, d, generator=gen).bfloat16().cuda() for _ in range(4)] for _ in range(2)]
    x = [torch.empty_like(t) for t in inputs[0]]
    out = [torch.empty(1, T, H, d, device="cuda") for _ in range(4)]

    def step():
        la.la_fwd_varlen(shape, *x[:3], LAM, out[0], cu, None, None, ws[0])
        la.la_bwd_varlen(shape, *x, LAM, *out[1:], cu, workspace=ws[1])

    want = []
    for given in inputs:
        for t, s in zip(x, given):
            t.copy_(s)
        step()
        want.append([t.clone() for t in out])
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        step()
    for w in ws:  # what an earlier call left is not what the replay reads
        w.zero_()
    for given, expect in zip(inputs, want):
        for t, s in zip(x, given):
            t.copy_(s)
        for t in out:
            t.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, expect))
    la.device_status()


@pytest.mark.parametrize("S", [333, 334, 2666, 2667, 5334])
def test_packed_tables_of_many_sequences(S):
    """The table goes in launches of up to 1000 or 8000 numbers, three for a sequence."""
    cu = np.concatenate([[0], np.cumsum(1 + np.arange(S) % 3)]).tolist()
    T = cu[-1]
    gen = torch.Generator().manual_seed(S)
    q, k, v = [torch.randn(1, T, 1, D, generator=gen).bfloat16().cuda() for _ in range(3)]
    shape = la.make_shape(1, 1, T, D, D, torch.bfloat16, torch.float32, layout=la.LA_LAYOUT_BNHD)
    o = torch.full((1, T, 1, D), float("nan"), device="cuda")
    ws = torch.empty(la.varlen_workspace_bytes(la.LA_OP_FWD, shape, cu), dtype=torch.uint8, device="cuda")
    n = la.launch_count()
    la.la_fwd_varlen(shape, q, k, v, torch.tensor([0.5]), o, cu, None, None, ws)
    assert la.launch_count() - n == 1
    torch.cuda.synchronize()
    la.device_status()
    # every sequence has up to three tokens: token t sees itself and the one or two before it in its sequence
    q, k, v = [t[0, :, 0].double().cpu() for t in (q, k, v)]
    want = torch.zeros(T, D, dtype=torch.float64)
    place = torch.arange(T) - torch.tensor(cu)[torch.searchsorted(torch.tensor(cu), torch.arange(T), right=True) - 1]
    for back in range(3):
        t = torch.nonzero(place >= back)[:, 0]
        want[t] += 0.5 ** back * (q[t] * k[t - back]).sum(1, keepdim=True) * v[t - back]
    rms = want.pow(2).mean().sqrt()
    assert (o[0, :, 0].double().cpu() - want).abs().max() <= 1.7e-4 * rms * 5  # (single rows reach several times the tensor's RMS)


@pytest.mark.parametrize("B,heads,N,segment", [
    (1, 8, 512, 512), (1, 8, 2048, 256), (1, 16, 8192, 1024), (1, 32, 777, 256), (1, 32, 1024, 256), (3, 16, 1536, 512),
    (4, 16, 1536, 1536), (4, 16, 1920, 1920), (4, 16, 2048, 1024), (4, 16, 16384, 8192)])
def test_segments_at_64_features(B, heads, N, segment):
    """The rule that its comment describes is the one that runs (the sizes are among those that were measured)."""
    assert la.segment_length(la.make_shape(B, heads, N, D, D, torch.bfloat16, torch.float32)) == segment


@pytest.mark.parametrize("lens,together", [([32768] + [100] * 10, False), ([8192] + [100] * 10, True), ([32768, 64], False)])
def test_packed_batches_of_uneven_lengths(lens, together):
    """One long sequence among short ones goes sequence by sequence, like the calls on each alone; others in one set of launches."""
    heads = 8
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    gen = torch.Generator("cuda")
    gen.manual_seed(7)
    q, k, v, do = [torch.randn(1, cu[-1], heads, D, generator=gen, device="cuda").bfloat16() for _ in range(4)]
    lam = torch.linspace(0.9, 1.0, heads)
    shape = la.make_shape(1, heads, cu[-1], D, D, torch.bfloat16, torch.float32, layout=la.LA_LAYOUT_BNHD)
    ws = [torch.empty(la.varlen_workspace_bytes(op, shape, cu), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    out = [torch.full(q.shape, float("nan"), device="cuda") for _ in range(4)]
    n = la.launch_count()
    la.la_fwd_varlen(shape, q, k, v, lam, out[0], cu, None, None, ws[0])
    assert (la.launch_count() - n <= 3) == together
    la.la_bwd_varlen(shape, q, k, v, do, lam, *out[1:], cu, workspace=ws[1])
    want = [torch.empty_like(t) for t in out]
    for a, b in zip(cu, cu[1:]):
        one = la.make_shape(1, heads, b - a, D, D, torch.bfloat16, torch.float32, layout=la.LA_LAYOUT_BNHD)
        x, y = [t[:, a:b] for t in (q, k, v, do)], [t[:, a:b] for t in want]
        w = [torch.empty(max(256, la.workspace_bytes(op, one)), dtype=torch.uint8, device="cuda") for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
        la.la_fwd(one, *x[:3], lam, y[0], workspace=w[0])
        la.la_bwd(one, *x, lam, *y[1:], workspace=w[1])
    torch.cuda.synchronize()
    la.device_status()
    for a, b in zip(out, want):
        if together:  # two-term operands, 2^-17 of each product, in other segments: each side as above
            assert (a - b).abs().max() <= 2 * 1.7e-4 * b.pow(2).mean().sqrt() * 5
        else:
            assert torch.equal(a, b)


@pytest.mark.parametrize("d", [64, 128])
def test_packed_calls_with_wrong_arguments_launch_nothing(d):
    cu = [0, 100, 300]
    shape = la.make_shape(1, H, cu[-1], d, d, torch.bfloat16, torch.float32, layout=la.LA_LAYOUT_BNHD)
    q, o = torch.zeros(1, cu[-1], H, d, device="cuda").bfloat16(), torch.zeros(1, cu[-1], H, d, device="cuda")
    ws = [torch.full((max(256, la.varlen_workspace_bytes(op, shape, cu)),), 7, dtype=torch.uint8, device="cuda")
          for op in (la.LA_OP_FWD, la.LA_OP_BWD)]
    wrong = torch.tensor([1.0, 2.0, 0.5])  # a rate above 1
    with pytest.raises(la.LaError):
        la.la_fwd_varlen(shape, q, q, q, wrong, o, cu, None, None, ws[0])
    with pytest.raises(la.LaError):
        la.la_bwd_varlen(shape, q, q, q, q, wrong, o, o.clone(), o.clone(), cu, workspace=ws[1])
    torch.cuda.synchronize()
    assert all(bool((w == 7).all()) for w in ws)
