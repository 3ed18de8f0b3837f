"""Performance cases of the M2RNN scan library: what its users run, through the public entry points.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

  token     one decoded token through a whole layer: conv (with the carried rows), decoding step on
            the cached state, gated norm -- what a chat session costs per layer and token
  decode    one decoding step of a serving batch on its cached states
  prompt    a prompt through a whole layer: conv over the fused projection, scan on column slices of
            the result (no copies), gated norm; the final state starts the decoding
  prefill   the scan alone, dense layout, keeping the final state
  train     the scan forward with checkpoints and its backward through time
  conv      forward and backward of the input path (conv + SiLU)
  norm      forward and backward of the output path (gated RMSNorm)

Shapes and distributions are those of the benchmark configurations (``inputs.CONFIGS``): q, k, v ~
N(0,1)/sqrt(K), logit gates ~ N(2,1), initial states ~ N(0, 0.1^2); whole layers take the paper's own
forget gate (``psi``).  W is the identity for V = 16, the state size of the paper's own layers, which
initialise it so, and else N(0, 0.5^2/V), a contracting map: with N(0, 1/V) some heads are chaotic
and no two implementations agree on their gradients (measured: two kernels of this library differ by
3e-3 to 0.8 there), which no training run could use either.  Everything is drawn on the GPU from the
seed.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2603_14360_b200 import binding as m

IO = {"bf16": torch.bfloat16, "f32": torch.float32}
SCAN = ("token", "decode", "prompt", "prefill", "train")


def listed():
    return [
        # one session, one token, the paper's layer (84 value heads share one q/k head): latency
        dict(name="token_layer", kind="token", dtype="bf16", B=1, T=1, N=84, shared=True, K=64, V=16),
        # a small serving batch on the same layer
        dict(name="decode_layer", kind="decode", dtype="bf16", B=48, T=1, N=84, shared=True, K=64, V=16),
        # the `decode` configuration: 512 sessions, large states, bound by HBM
        dict(name="decode_full", kind="decode", dtype="bf16", B=512, T=1, N=32, shared=False, K=128, V=128),
        # a prompt of odd length through the paper's layer
        dict(name="prompt_layer", kind="prompt", dtype="bf16", B=1, T=1001, N=84, shared=True, K=64, V=16),
        # the `fwd_bf16` configuration
        dict(name="prefill_batch", kind="prefill", dtype="bf16", B=8, T=2048, N=16, shared=False, K=64, V=64),
        # the `long_ctx` configuration: one very long sequence
        dict(name="prefill_long", kind="prefill", dtype="bf16", B=1, T=65536, N=32, shared=False, K=128, V=128),
        # the paper's layer at its training context (`paper_layer`)
        dict(name="train_layer", kind="train", dtype="bf16", B=4, T=4096, N=84, shared=True, K=64, V=16, packed=False),
        # the `bptt_bf16` configuration
        dict(name="train_batch", kind="train", dtype="bf16", B=8, T=4096, N=32, shared=False, K=64, V=64, packed=False),
        # documents of ragged lengths packed into one batch, q/k/v slices of a fused projection, the
        # largest state of the state-size sweep
        dict(name="train_packed", kind="train", dtype="bf16", B=12, T=4000, N=16, shared=False, K=128, V=128, packed=True),
        # fp32, the accuracy path: a small model checked or trained in full precision
        dict(name="train_f32", kind="train", dtype="f32", B=2, T=512, N=8, shared=False, K=64, V=64, packed=False),
        # the input path on the fused projection of `fwd_bf16`
        dict(name="conv_batch", kind="conv", dtype="bf16", B=8, T=2048, C=3072),
        # the output path on the tokens of `paper_layer`: rows of 84 x 16 features
        dict(name="norm_layer", kind="norm", dtype="bf16", B=4, T=4096, N=84, V=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(case):
    """Serial length of a scan in forward steps at V = 128: T times the waves its 16-row slabs (fp32:
    its units) need, times what a backward and an fp32 step cost against that."""
    units = case["B"] * case["N"]
    if case["dtype"] == "f32":
        return case["T"] * -(-units // 148) * (160 if case["kind"] == "train" else 40) * max(0.25, case["K"] * case["V"] ** 2 / 64 ** 3)
    waves = -(-units * case["K"] // 16 // 592)
    return case["T"] * waves * (5 if case["kind"] == "train" else 1) * max(case["V"], 32) / 128


def draw(rng):
    top = work(listed()[5])
    while True:
        kind = rng.choice(("token", "decode", "decode", "prompt", "prefill", "prefill", "train", "train", "train", "conv", "norm"))
        case = dict(kind=kind, dtype="f32" if rng.random() < 0.15 else "bf16")
        if kind == "conv":
            case.update(B=rng.randint(1, 8), T=_log(rng, 16, 8192), C=8 * _log(rng, 16, 1024))
        elif kind == "norm":
            case.update(B=rng.randint(1, 8), T=_log(rng, 16, 8192), N=rng.randint(4, 96), V=rng.choice((16, 32, 64)))
        else:
            V = rng.choice((16, 32, 64, 128))
            K = 64 if V == 16 and rng.random() < 0.5 else V if rng.random() < 0.6 else 16 * rng.randint(1, 8)
            B = {"token": rng.randint(1, 8), "decode": _log(rng, 1, 512), "prompt": rng.randint(1, 4)}.get(kind) or _log(rng, 1, 16)
            T = {"token": 1, "decode": 1, "prompt": _log(rng, 16, 8192), "prefill": _log(rng, 16, 65536), "train": _log(rng, 32, 8192)}[kind]
            case.update(B=B, T=T, N=rng.randint(2, 96), shared=V == 16 or rng.random() < 0.3, K=K, V=V)
            if kind == "train":
                case.update(packed=rng.random() < 0.3)
            if _steps(case) > 65536:
                continue
        w = work(case)
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"]:
            return case


def _lengths(case):
    """Token counts of the documents of a packed batch; the longest is T."""
    rng = random.Random(1000003 * case["T"] + 101 * case["B"] + case["N"])
    return [case["T"]] + [max(1, int(case["T"] * rng.uniform(0.02, 1.0) ** 1.5)) for _ in range(case["B"] - 1)]


def _tokens(case):
    return sum(_lengths(case)) if case.get("packed") else case["B"] * case["T"]


def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    tok, kind = _tokens(case), case["kind"]
    if kind == "conv":      # x, dout read, out, dx written; taps, bias and their sums
        return {"bytes": 4 * tok * case["C"] * e + case["C"] * (5 * e + 20), "flops": 34 * tok * case["C"]}
    if kind == "norm":      # y, g, dout read, out, dy, dg written; rstd
        d = case["N"] * case["V"]
        return {"bytes": 6 * tok * d * e + 4 * tok + d * (e + 4), "flops": 30 * tok * d}
    N, K, V = case["N"], case["K"], case["V"]
    h = 1 if case["shared"] else N
    states = case["B"] * N * K * V * 4
    qkv, W, y = tok * (2 * h * K + N * V) * e, N * V * V * e, tok * N * V * e
    flops = tok * N * (2 * K * V * V + 4 * K * V)
    if kind in ("token", "decode", "prefill"):   # the state is read once and written once
        extra = 0
        if kind == "token":     # projections and gate input read, normalised row written, taps, bias, carried rows
            C = 2 * h * K + N * V
            extra = tok * N * V * e + (C * 5 + 3 * C * case["B"] + N * V) * e
        return {"bytes": qkv + W + y + tok * N * 4 + 2 * states + extra, "flops": flops}
    if kind == "prompt":        # no initial state; the final one is written
        C = 2 * h * K + N * V
        return {"bytes": qkv + W + y + tok * N * 4 + states + tok * N * V * e + (C * 5 + N * V) * e, "flops": flops + 9 * tok * C + 8 * tok * N * V}
    # train: q, k, v, gate, W, h0, dy read; y, hT, dq, dk, dv, dgate, dW, dh0 written
    return {"bytes": 2 * qkv + W + N * V * V * 4 + 2 * y + tok * N * 8 + 3 * states, "flops": 3 * flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5} if case["kind"] in ("conv", "norm") else {"rel": 5e-5, "max": 5e-3}
    if case["kind"] in ("conv", "norm", "token", "decode"):     # one rounding to bf16 each way
        return {"rel": 5e-3, "max": 5e-2}
    # bf16 operands and tanh.approx at every one of many steps of a recurrence
    return {"rel": 1e-2, "max": 0.2}


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(int(seed))
    io = IO[case["dtype"]]

    def normal(*shape, std=1.0, mean=0.0, to=io):
        return torch.empty(shape, dtype=to, device="cuda").normal_(mean, std, generator=gen)

    def uniform(*shape, lo, hi, to=io):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(lo, hi, generator=gen).to(to)

    B, T, kind = case["B"], case["T"], case["kind"]
    s = {"kind": kind}
    if kind == "conv":
        C = case["C"]
        s.update(x=normal(B, T, C), w=normal(C, 4, std=0.5), bias=normal(C, std=0.1), dout=normal(B, T, C))
        return s
    N, V = case["N"], case["V"]
    if kind == "norm":
        s.update(y=normal(B, T, N, V), g=normal(B, T, N, V), w=uniform(N * V, lo=0.5, hi=1.5), dout=normal(B, T, N, V))
        return s
    K = case["K"]
    h = 1 if case["shared"] else N
    std = K ** -0.5
    s["W"] = torch.eye(V, device="cuda").expand(N, V, V).to(io).contiguous() if V == 16 else normal(N, V, V, std=0.5 * V ** -0.5)
    f32 = torch.float32
    if kind in ("token", "prompt"):
        C = 2 * h * K + N * V
        s.update(x=normal(B, T, C), conv_w=normal(C, 4, std=0.5), bias=normal(C, std=0.1), g=normal(B, T, N, V), norm_w=uniform(N * V, lo=0.5, hi=1.5),
                 gate=normal(B, T, N, mean=-3.0, to=f32), alpha=uniform(N, lo=0.5, hi=2.0, to=f32), beta=uniform(N, lo=0.1, hi=2.0, to=f32),
                 prev=normal(B, 3, C) if kind == "token" else None, split=(h * K, 2 * h * K), heads=h, N=N)
        if kind == "token":
            s["state"] = normal(B, N, K, V, std=0.1, to=f32)
        return s
    if kind == "decode":
        s.update(q=normal(B, h, K, std=std), k=normal(B, h, K, std=std), v=normal(B, N, V, std=std), gate=normal(B, N, mean=2.0, to=f32),
                 state=normal(B, N, K, V, std=0.1, to=f32))
        return s
    s["more"] = {}
    if case.get("packed"):
        lens = _lengths(case)
        lead = (sum(lens),)
        cu = torch.zeros(B + 1, dtype=torch.int32)
        cu[1:] = torch.tensor(lens, dtype=torch.int32).cumsum(0)
        s["more"] = dict(cu_seqlens=cu.cuda(), max_seqlen=T)
        fused = normal(lead[0], 2 * h * K + N * V, std=std)     # one projection output, used through its slices
        s.update(q=fused[:, : h * K].unflatten(1, (h, K)), k=fused[:, h * K: 2 * h * K].unflatten(1, (h, K)),
                 v=fused[:, 2 * h * K:].unflatten(1, (N, V)))
    else:
        lead = (B, T)
        s.update(q=normal(B, T, h, K, std=std), k=normal(B, T, h, K, std=std), v=normal(B, T, N, V, std=std))
    s.update(gate=normal(*lead, N, mean=2.0, to=f32), h0=normal(B, N, K, V, std=0.1, to=f32))
    if kind == "train":
        s["dy"] = normal(*lead, N, V)
    return s


def run(s):
    kind = s["kind"]
    if kind == "conv":
        out = m.m2rnn_conv_silu_fwd(s["x"], s["w"], s["bias"])
        g = m.m2rnn_conv_silu_bwd(s["x"], s["w"], s["dout"], s["bias"])
        return out, g["dx"], g["dw"], g["dbias"]
    if kind == "norm":
        out, rstd = m.m2rnn_gated_norm_fwd(s["y"], s["g"], s["w"], eps=1e-6)
        return out, m.m2rnn_gated_norm_bwd(s["y"], s["g"], s["w"], rstd, s["dout"])
    if kind == "decode":
        return m.m2rnn_decode_step(s["q"], s["k"], s["v"], s["gate"], s["W"], s["state"]), s["state"]
    if kind == "prefill":
        y, hT, _ = m.m2rnn_fwd(s["q"], s["k"], s["v"], s["gate"], s["W"], s["h0"])
        return y, hT
    if kind == "train":
        y, hT, ckpt = m.m2rnn_fwd(s["q"], s["k"], s["v"], s["gate"], s["W"], s["h0"], save_ckpt=True, **s["more"])
        return y, hT, m.m2rnn_bwd(s["q"], s["k"], s["v"], s["gate"], s["W"], s["h0"], s["dy"], ckpt=ckpt, **s["more"])
    # a whole layer between its projections
    psi = dict(gate_kind=m.GATE_PSI, alpha=s["alpha"], beta=s["beta"])
    c = m.m2rnn_conv_silu_fwd(s["x"], s["conv_w"], s["bias"], s["prev"])
    (i, j), h, N = s["split"], s["heads"], s["N"]
    q, k, v = c[:, :, :i].unflatten(2, (h, -1)), c[:, :, i:j].unflatten(2, (h, -1)), c[:, :, j:].unflatten(2, (N, -1))
    if kind == "prompt":
        y, hT, _ = m.m2rnn_fwd(q, k, v, s["gate"], s["W"], **psi)
    else:       # the decoding step takes dense rows
        y, hT = m.m2rnn_decode_step(q[:, 0].contiguous(), k[:, 0].contiguous(), v[:, 0].contiguous(), s["gate"][:, 0], s["W"], s["state"], **psi)[:, None], s["state"]
    return m.m2rnn_gated_norm_fwd(y, s["g"], s["norm_w"], eps=1e-6)[0], hT
