"""The work that is timed: calls of the library's public entry points (paper_2307_14995_b200.binding) as a program that
trains or serves the model makes them.

Five kinds of calls stand for five uses:

  train    la_fwd then la_bwd on the workspace the forward pass left: one layer's token mixer in a training step
  mixer    la_fwd_gated (keeping o), la_gate_bwd, la_bwd: the same with the output stage y = SRMSNorm(o) (.) u
  lrpe     la_lrpe_fwd then la_lrpe_bwd: the layer with the learnable rotation
  prefill  la_fwd with the state handed in and out: a prompt, or one chunk of a prompt, before decoding
  packed   la_fwd_varlen (and la_bwd_varlen when training): sequences of different lengths in one packed tensor
  decode   la_decode_step / la_decode_steps on a state that is updated in place: one token, or a few drafted ones

Values are drawn as the token mixer sees them: q, k = SiLU(N(0,1)), v, dO, u ~ N(0,1), and one decay rate per head from
the layer's position in the model.  Everything is made on the GPU from the seed.
"""
import torch

from paper_2307_14995_b200 import binding as la, inputs

_DTYPE = {"bf16": torch.bfloat16, "fp32": torch.float32}
_BYTES = {"bf16": 2, "fp32": 4}
_LAYOUT = {"heads": la.LA_LAYOUT_BHND, "tokens": la.LA_LAYOUT_BNHD}


def _case(kind, B, H, N, d, **more):
    c = {"kind": kind, "B": B, "H": H, "N": N, "d": d, "inp": "bf16", "out": "fp32", "layout": "heads", "depth": 0.5}
    c.update(more)
    return c


def listed():
    cases = [
        # the fp32 reference configuration: the smallest training call, through the wrappers that allocate their outputs
        ("train_fp32_ref", _case("train", 1, 2, 256, 64, inp="fp32", wrapped=True)),
        # one training step of a layer of the 385M-like, the 1B-like and the long-context 7B-like configuration
        ("train_385m", _case("train", 4, 16, 2048, 64, depth=0.25)),
        ("train_1b", _case("train", 2, 16, 8192, 128)),
        ("train_7b_long", _case("train", 1, 32, 65536, 128, depth=0.9)),
        # mixed-precision training as a projection hands it over: token-major, bf16 results, a length of no round size
        ("train_bf16_ragged", _case("train", 3, 8, 3001, 128, out="bf16", layout="tokens")),
        # the token mixer with its output stage, forward and backward, 1B-like
        ("mixer_1b", _case("mixer", 2, 16, 8192, 128)),
        # the first layer's variant with the learnable rotation
        ("lrpe_1b", _case("lrpe", 1, 16, 8192, 128, depth=0.0)),
        # serving: a short prompt continuing an earlier state, and many prompts packed together
        ("prefill_short", _case("prefill", 1, 32, 777, 128, out="bf16", layout="tokens", depth=0.9)),
        ("prefill_packed", _case("packed", 48, 32, 3000, 128, depth=0.9, backward=False)),
        # serving: a single conversation, a full batch, and drafted tokens checked together
        ("decode_single", _case("decode", 1, 32, 1, 128, out="bf16", depth=0.9)),
        ("decode_batch64", _case("decode", 64, 32, 1, 128, depth=0.9)),
        ("decode_draft", _case("decode", 16, 32, 4, 128, out="bf16", depth=0.9)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, low, high):
    return int(round(low * (high / low) ** rng.random()))


def draw(rng):
    kind = rng.choice(("train", "train", "train", "mixer", "lrpe", "prefill", "packed", "decode"))
    d = rng.choice((64, 128, 128))
    H = rng.choice((8, 16, 32))
    depth = rng.choice((0.0, 0.25, 0.5, 0.9, 1.0))
    form = {"out": rng.choice(("fp32", "bf16")), "layout": rng.choice(("heads", "tokens")), "depth": depth}
    if kind == "decode":
        return _case(kind, _log_int(rng, 1, 128), H, rng.choice((1, 1, 1, 2, 3, 4, 8)), d, **form)
    if kind == "packed":
        form.update(layout="tokens", backward=rng.random() < 0.5)
        return _case(kind, _log_int(rng, 2, 64), H, _log_int(rng, 100, 4096), d, **form)
    if kind == "prefill":
        return _case(kind, _log_int(rng, 1, 8), H, _log_int(rng, 16, 16384), d, **form)
    if kind == "lrpe":
        return _case(kind, rng.choice((1, 2)), H, _log_int(rng, 256, 8192), d, **form)
    if kind == "mixer":
        B = rng.choice((1, 2, 4))
        return _case(kind, B, H, _log_int(rng, 256, 32768 // B), d, **form)
    if rng.random() < 0.25:  # full precision: checks and small models
        form.update(inp="fp32", out="fp32")
        return _case(kind, rng.choice((1, 2)), rng.choice((2, 4, 8)), _log_int(rng, 64, 2048), d, **form)
    B = rng.choice((1, 1, 2, 4))
    return _case(kind, B, H, _log_int(rng, 128, 65536 // B), d, **form)


def _lengths(case):
    """The packed batch's sequence lengths: between an eighth of N and N, with odd ones among them; the same for every seed."""
    S, N = case["B"], case["N"]
    low = max(1, N // 8)
    return [low + (i * 7919 + 13) % (N - low + 1) for i in range(S)]


def _tokens(case):
    return sum(_lengths(case)) if case["kind"] == "packed" else case["B"] * case["N"]


def prepare(case, seed):
    kind, B, H, N, d = (case[x] for x in ("kind", "B", "H", "N", "d"))
    inp, out, layout = _DTYPE[case["inp"]], _DTYPE[case["out"]], _LAYOUT[case["layout"]]
    dev = torch.device("cuda")
    gen = torch.Generator(dev)
    gen.manual_seed(seed)
    if kind == "packed":
        B, N, layout = 1, _tokens(case), la.LA_LAYOUT_BNHD
    size = (B, N, H, d) if layout == la.LA_LAYOUT_BNHD else (B, H, N, d)
    scale = d ** -0.5 if case["inp"] == "fp32" else 1.0  # as the fp32 reference configuration draws q and k

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    def silu(*shape):
        return (torch.nn.functional.silu(normal(*shape)) * scale).to(inp)

    def empty(*shape, dtype=out):
        return torch.empty(shape, dtype=dtype, device=dev)

    s = {"kind": kind, "lam": inputs.decay_rates(H, case["depth"]), "shape": la.make_shape(B, H, N, d, d, inp, out, layout=layout)}
    s["q"], s["k"], s["v"] = silu(*size), silu(*size), normal(*size).to(inp)
    s["o"] = empty(*size)
    shape = s["shape"]
    if kind == "decode":
        # the state an earlier prompt of 64 tokens left
        past_k, past_v = torch.nn.functional.silu(normal(B, H, 64, d)), normal(B, H, 64, d)
        age = torch.arange(63, -1, -1, device=dev, dtype=torch.float32)
        past_k *= s["lam"].to(dev).view(1, H, 1, 1) ** age.view(1, 1, 64, 1)
        s["kv"] = torch.matmul(past_k.transpose(2, 3), past_v).contiguous()
        return s
    if kind == "prefill":
        s["kv_in"], s["kv_out"] = 4 * normal(B, H, d, d), empty(B, H, d, d, dtype=torch.float32)
        s["ws_f"] = la.alloc_workspace(la.LA_OP_FWD, shape, dev)
        return s
    if kind == "packed":
        cu = [0]
        for n in _lengths(case):
            cu.append(cu[-1] + n)
        s["cu"], s["backward"] = cu, case["backward"]
        s["kv_out"] = empty(case["B"], H, d, d, dtype=torch.float32)
        s["ws_f"] = empty(max(256, la.varlen_workspace_bytes(la.LA_OP_FWD, shape, cu)), dtype=torch.uint8)
        if not case["backward"]:
            return s
        s["ws_b"] = empty(max(256, la.varlen_workspace_bytes(la.LA_OP_BWD, shape, cu)), dtype=torch.uint8)
    s["do"] = normal(*size).to(inp)
    if case.get("wrapped"):
        s["kind"], s["out_dtype"] = "wrapped", out
        return s
    s["dq"], s["dk"], s["dv"] = empty(*size), empty(*size), empty(*size)
    if kind == "lrpe":
        s["theta"] = inputs.make_theta(H, d, seed=seed).to(dev)
        s["dtheta"] = empty(H, d, dtype=torch.float32)
        s["ws_f"] = empty(la.lrpe_workspace_bytes(la.LA_OP_FWD, shape), dtype=torch.uint8)
        s["ws_b"] = empty(la.lrpe_workspace_bytes(la.LA_OP_BWD, shape), dtype=torch.uint8)
        return s
    if kind == "mixer":
        s["u"], s["y"] = normal(*size).to(inp), empty(*size)
        s["d_o"], s["du"] = empty(*size, dtype=inp), empty(*size)
    if kind != "packed":
        s["ws_f"] = la.alloc_workspace(la.LA_OP_FWD, shape, dev)
        s["ws_b"] = la.alloc_workspace(la.LA_OP_BWD, shape, dev)
    return s


def run(s):
    kind, shape, lam, q, k, v = (s[x] for x in ("kind", "shape", "lam", "q", "k", "v"))
    if kind == "decode":
        if shape.N == 1:
            la.la_decode_step(shape, q, k, v, lam, s["kv"], s["o"])
        else:
            la.la_decode_steps(shape, q, k, v, lam, s["kv"], s["o"])
        return s["o"], s["kv"]
    if kind == "prefill":
        la.la_fwd(shape, q, k, v, lam, s["o"], s["kv_in"], s["kv_out"], s["ws_f"])
        return s["o"], s["kv_out"]
    if kind == "packed":
        la.la_fwd_varlen(shape, q, k, v, lam, s["o"], s["cu"], None, s["kv_out"], s["ws_f"])
        if not s["backward"]:
            return s["o"], s["kv_out"]
        la.la_bwd_varlen(shape, q, k, v, s["do"], lam, s["dq"], s["dk"], s["dv"], s["cu"], workspace=s["ws_b"])
        return s["o"], s["kv_out"], s["dq"], s["dk"], s["dv"]
    if kind == "wrapped":
        o = la.fwd(q, k, v, lam, out_dtype=s["out_dtype"])
        return (o,) + la.bwd(q, k, v, s["do"], lam, out_dtype=s["out_dtype"])
    o, do, dq, dk, dv = s["o"], s["do"], s["dq"], s["dk"], s["dv"]
    if kind == "lrpe":
        la.la_lrpe_fwd(shape, q, k, v, s["theta"], lam, o, workspace=s["ws_f"])
        la.la_lrpe_bwd(shape, q, k, v, do, s["theta"], lam, dq, dk, dv, s["dtheta"], workspace=s["ws_b"])
        return o, dq, dk, dv, s["dtheta"]
    if kind == "mixer":
        la.la_fwd_gated(shape, q, k, v, s["u"], lam, s["y"], o, workspace=s["ws_f"])
        la.la_gate_bwd(shape, o, s["u"], do, s["d_o"], s["du"])
        la.la_bwd(shape, q, k, v, s["d_o"], lam, dq, dk, dv, workspace=s["ws_b"], fwd_workspace=s["ws_f"])
        return s["y"], o, s["du"], dq, dk, dv
    la.la_fwd(shape, q, k, v, lam, o, workspace=s["ws_f"])
    la.la_bwd(shape, q, k, v, do, lam, dq, dk, dv, workspace=s["ws_b"], fwd_workspace=s["ws_f"])
    return o, dq, dk, dv


def work(case):
    """Every input read once and every output written once; flops of the block method with 128-token blocks (half of
    each score tile), or of the token recurrence where that is what a call runs."""
    kind, H, d = case["kind"], case["H"], case["d"]
    rows = _tokens(case) * H                       # (token, head) pairs
    i, o = _BYTES[case["inp"]], _BYTES[case["out"]]
    fwd, bwd = 2 * 128 * d + 4 * d * d, 5 * 128 * d + 10 * d * d
    state = H * d * d * 4
    if kind == "decode":
        return {"bytes": 2 * case["B"] * state + rows * d * (3 * i + o), "flops": rows * 5 * d * d}
    if kind == "prefill":
        return {"bytes": 2 * case["B"] * state + rows * d * (3 * i + o), "flops": rows * fwd}
    if kind == "packed" and not case["backward"]:
        return {"bytes": case["B"] * state + rows * d * (3 * i + o), "flops": rows * fwd}
    step = {"bytes": rows * d * (4 * i + 4 * o), "flops": rows * (fwd + bwd)}
    if kind == "packed":
        step["bytes"] += case["B"] * state
    elif kind == "mixer":                          # u besides, and y and du
        step["bytes"] += rows * d * (i + 2 * o)
        step["flops"] += rows * 15 * d
    elif kind == "lrpe":                           # the score and the state have two parts, one per rotated feature
        step["bytes"] += 2 * H * d * 4
        step["flops"] = rows * (3 * 128 * d + 8 * d * d + 8 * 128 * d + 20 * d * d)
    return step


def tolerance(case):
    """About four times the largest difference from the same path in 64 bits (d = 64 and 128, all depths, 777 to 2048
    tokens; relative 2-norm, then largest difference)."""
    bf16_out = case["out"] == "bf16"
    if case["kind"] == "mixer":    # d_o between the two passes is rounded to bf16: 3.1e-3 (fp32 results), 4.4e-3
        return {"rel": 1.7e-2 if bf16_out else 1.2e-2}
    if case["kind"] == "lrpe":     # the rotated features are rounded to bf16: 3.1e-3 and 3.9e-3, largest 2.3e-2
        return {"rel": 1.6e-2 if bf16_out else 1.2e-2, "max": 0.1}
    if bf16_out:                   # the rounding of the results: 1.7e-3, largest 3.9e-3
        return {"rel": 7e-3, "max": 1.6e-2}
    if case["kind"] == "decode":   # fp32 sums: 8e-8, largest 4.4e-7
        return {"rel": 5e-7, "max": 4e-6}
    if case["inp"] == "fp32":      # fp32 sums: 2.0e-7, largest 2.2e-6
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 1e-5, "max": 2e-4}  # two-term bf16 operands: 2.5e-6, largest 4.3e-5
