"""Backward scan of V = 16 problems with more slabs of 16 rows than SMs (scan_bwd_v16.cu) against the fp64 oracle: CTAs of
several heads and slabs, shares of shared heads, ragged chunks, every checkpoint interval's kind.  Bound: the bf16 path's 2e-2
(parity.TOL); two forms of the same sums: the order of at most 128 fp32 terms."""
import ctypes
import dataclasses
import os
import subprocess
import sys

import pytest
import torch

import parity
from paper_2603_14360_b200 import binding, inputs
from paper_2603_14360_b200.inputs import GATE_LOGIT, GATE_PSI, GATE_VALUE, ScanConfig

# B, T, N, K, Nq, Nk
SHAPES = [
    (2, 33, 84, 64, 1, 1),       # the paper's layer: heads in pieces of several, the last piece shorter
    (4, 17, 21, 48, 1, 1),       # three slabs a state; a prime number of heads
    (8, 9, 20, 16, 20, 20),      # one slab a state, a q and a k head each
    (3, 26, 12, 128, 1, 12),     # eight slabs; q shared, k not
    (3, 23, 12, 80, 12, 2),      # five slabs; k shared by two sets, q not
    (2, 8, 24, 96, 2, 3),        # sets of four heads: the largest that share both
    (40, 1, 4, 64, 2, 2),        # a single step; whole sets in a CTA: no shares
    (6, 19, 10, 112, 1, 1),      # seven slabs
]


def _cfg(shape, gate_kind=GATE_LOGIT, **kw):
    B, T, N, K, Nq, Nk = shape
    return ScanConfig("v16", B=B, T=T, N=N, K=K, V=16, Nq=Nq, Nk=Nk, gate_kind=gate_kind, gate_mean=1.0,
                      w_scale=0.5 if gate_kind == GATE_PSI else 1.0, seed=400 + T, **kw)


@pytest.mark.gpu
@pytest.mark.parametrize("gate_kind", [GATE_VALUE, GATE_LOGIT, GATE_PSI])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_shapes(oracle, shape, gate_kind):
    assert shape[0] * shape[2] * shape[3] // 16 > 148
    parity.check_bwd(oracle, _cfg(shape, gate_kind), residual=True, d_hT=True)


@pytest.mark.gpu
@pytest.mark.parametrize("C", [2, 6, 8, 10, 16])
def test_intervals(oracle, C):
    cfg = _cfg((4, 37, 12, 64, 1, 1))
    d = inputs.make_inputs(cfg, backward=True)
    ref, g = parity.oracle_bwd(oracle, cfg, d), parity.to_dev(d)
    for ckpt in (parity.gpu_fwd(cfg, g, save_ckpt=True, ckpt_interval=C)[2], None):
        out = parity.gpu_bwd(cfg, g, ckpt=ckpt, ckpt_interval=C)
        binding.check_device_status()
        for name in ref:
            assert parity.rel_err(out[name], ref[name]) <= parity.TOL["bf16"], (C, name)


# sizes whose checkpoints come every eight steps and whose chunks, from some T on, have sixteen
TWO = [(3, 12, 128, 1, 12), (2, 84, 64, 1, 1)]      # B, N, K, Nq, Nk


@pytest.mark.gpu
@pytest.mark.parametrize("T,size", [(26, TWO[0]), (40, TWO[0]), (47, TWO[0]), (200, TWO[1])], ids=str)
def test_chunks_of_two_intervals(oracle, T, size):
    """A ragged last chunk of one and of two checkpoints; the call's own checkpoints too, and every second one asked for by the caller."""
    B, N, K, Nq, Nk = size
    # (a contracting W: with N(0, 1/V) some heads amplify a rounding over 200 steps, and two forms of the same kernel differ by 4e-2)
    cfg = dataclasses.replace(_cfg((B, T, N, K, Nq, Nk)), w_scale=0.5)
    p = binding.Params(B=B, T=T, N=N, Nq=Nq, Nk=Nk, K=K, V=16, io_dtype=1, gate_kind=1, ckpt_interval=0, dh_clip=0.0)
    assert binding.m2rnn_ckpt_interval(p) == 8 and binding.m2rnn_bwd_row_slab(p) == 16
    d = inputs.make_inputs(cfg, backward=True, d_hT=True)
    ref, g = parity.oracle_bwd(oracle, cfg, d), parity.to_dev(d)
    ckpt = parity.gpu_fwd(cfg, g, save_ckpt=True)[2]
    assert ckpt.shape[2] == -(-T // 8)
    for kw in (dict(ckpt=ckpt), dict(), dict(ckpt=ckpt[:, :, ::2].contiguous(), ckpt_interval=16)):
        out = parity.gpu_bwd(cfg, g, **kw)
        binding.check_device_status()
        for name in ref:
            assert parity.rel_err(out[name], ref[name]) <= parity.TOL["bf16"], (list(kw), name)


@pytest.mark.gpu
def test_chunks_of_two_intervals_clipped(oracle):
    B, N, K, Nq, Nk = TWO[0]
    parity.check_bwd(oracle, ScanConfig("clip", B=B, T=40, N=N, K=K, V=16, Nq=Nq, Nk=Nk, dist="saturating", gate_mean=1.0, seed=9), dh_clip=0.5)


@pytest.mark.gpu
def test_chunks_of_two_intervals_packed():
    """Sequences that end in every part of a chunk, an empty one among them: as each by itself."""
    (B, N, K, Nq, Nk), lens = TWO[0], [41, 0, 8, 25, 16, 1]
    tok, gen = sum(lens), torch.Generator("cuda").manual_seed(6)
    rnd = lambda *s, dt=torch.bfloat16, std=1.0: torch.empty(s, dtype=dt, device="cuda").normal_(0, std, generator=gen)
    q, k, v = rnd(tok, Nq, K, std=0.125), rnd(tok, Nk, K, std=0.125), rnd(tok, N, 16)
    gate, W, dy, h0 = rnd(tok, N, dt=torch.float32), rnd(N, 16, 16, std=0.125), rnd(tok, N, 16), rnd(len(lens), N, K, 16, dt=torch.float32, std=0.1)
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0, dtype=torch.int32).cuda()
    pk = dict(cu_seqlens=cu, max_seqlen=max(lens))
    ckpt = binding.m2rnn_fwd(q, k, v, gate, W, h0, save_ckpt=True, **pk)[2]
    got = binding.m2rnn_bwd(q, k, v, gate, W, h0, dy, ckpt=ckpt, **pk)
    at = 0
    for b, n in enumerate(lens):
        sl, at = slice(at, at + n), at + n
        if n:
            one = binding.m2rnn_bwd(*(x[None, sl].contiguous() for x in (q, k, v, gate)), W, h0[b:b + 1], dy[None, sl])
            for name in ("dq", "dk", "dv", "dgate"):
                assert parity.rel_err(got[name][sl], one[name][0].double().cpu().numpy()) < 2.0 ** -8, (b, name)     # (a rounding to bf16)
    binding.check_device_status()


@pytest.mark.gpu
def test_clipping(oracle):
    parity.check_bwd(oracle, ScanConfig("clip", B=4, T=24, N=12, K=64, V=16, dist="saturating", gate_mean=1.0, seed=9), dh_clip=0.5)


@pytest.mark.gpu
def test_packed_slices_match_the_sequences_one_by_one(oracle):
    """Ragged sequences, an empty one among them, q/k/v slices of one tensor: as each sequence by itself."""
    lens, N, K, f32 = [19, 0, 1, 40, 8], 16, 64, torch.float32
    gen = torch.Generator("cuda").manual_seed(5)
    rnd = lambda *s, dt=torch.bfloat16, std=1.0: torch.empty(s, dtype=dt, device="cuda").normal_(0, std, generator=gen)
    tok = sum(lens)
    fused = rnd(tok, 2 * K + N * 16, std=0.125)
    q, k, v = fused[:, :K].unflatten(1, (1, K)), fused[:, K:2 * K].unflatten(1, (1, K)), fused[:, 2 * K:].unflatten(1, (N, 16))
    gate, W, dy = rnd(tok, N, dt=f32), rnd(N, 16, 16, std=0.125), rnd(tok, N, 16)
    h0, d_hT = rnd(len(lens), N, K, 16, dt=f32, std=0.1), rnd(len(lens), N, K, 16, dt=f32)
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0, dtype=torch.int32).cuda()
    got = binding.m2rnn_bwd(q, k, v, gate, W, h0, dy, d_hT, cu_seqlens=cu, max_seqlen=max(lens))
    dW, at = torch.zeros_like(got["dW"]), 0
    for b, n in enumerate(lens):
        if n == 0:
            assert torch.equal(got["dh0"][b], d_hT[b])
            continue
        sl = slice(at, at + n)
        one = binding.m2rnn_bwd(*(x[None, sl].contiguous() for x in (q, k, v, gate)), W, h0[b:b + 1], dy[None, sl], d_hT[b:b + 1])
        for name in ("dq", "dk", "dv", "dgate"):
            assert parity.rel_err(got[name][sl], one[name][0].double().cpu().numpy()) < 2.0 ** -8, (b, name)     # (a rounding to bf16)
        assert parity.rel_err(got["dh0"][b], one["dh0"][0].double().cpu().numpy()) < 1e-5
        dW, at = dW + one["dW"], at + n
    binding.check_device_status()
    assert parity.rel_err(got["dW"], dW.double().cpu().numpy()) < 1e-5


def test_limited_scratch_holds_the_calls_own_checkpoints():
    """Nothing asks for checkpoints every eight steps where the call makes its own and its chunks have sixteen: 7.0 to 7.9 MiB, and 2.3 to
    3.4 more with twice as many (-6: accepted, and no device)."""
    code = ("import ctypes, sys; sys.path[:0] = [%r]\n"
            "from paper_2603_14360_b200 import build, binding as b\n"
            "build.build()\n"
            "f = ctypes.c_void_p(0x10000)\n"
            "for B, T, N, Nq in ((6, 100, 8, 1), (6, 144, 8, 4), (2, 256, 12, 6)):\n"
            "    p = b.Params(B=B, T=T, N=N, Nq=Nq, Nk=1, K=128, V=16, io_dtype=1, gate_kind=1, ckpt_interval=0, dh_clip=0.0)\n"
            "    print(b._lib().m2rnn_ckpt_interval(ctypes.byref(p)),\n"
            "          b._lib().m2rnn_bwd_static_scratch(ctypes.byref(p), *([f] * 5), None, None, None, None, None, f, None, *([f] * 5), None, None, None))\n"
            ) % os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}, timeout=300)
    assert r.stdout.split() == ["8", "-6"] * 3, (r.stdout, r.stderr[-2000:])


def test_scratch_where_it_is_limited():
    """No more scratch than a share of dq and dk per head and of dv, dgate and dW per CTA of `rows` rows; m2rnn_bwd_static_scratch takes
    what fits with checkpoints every 16 steps and as many rows and heads a CTA as there can be (-6: accepted, and no device)."""
    from paper_2603_14360_b200 import build
    build.build()
    lib = binding._lib()
    P = lambda **kw: binding.Params(**{**dict(B=2, T=64, N=84, Nq=1, Nk=1, K=64, V=16, io_dtype=1, gate_kind=1, ckpt_interval=0, dh_clip=0.0), **kw})
    for B, T, N, K in ((2, 16, 84, 64), (3, 24, 50, 96), (4, 64, 16, 64), (16, 16, 21, 16)):
        p = P(B=B, T=T, N=N, K=K)
        rows = lib.m2rnn_bwd_row_slab(ctypes.byref(p))
        assert K % rows == 0 and rows % 16 == 0
        RS = K // rows
        most = 4 * (2 * B * T * N * K + B * RS * N * 256 + (RS > 1) * RS * B * T * N * 17) + 8 * 256
        assert lib.m2rnn_bwd_workspace_bytes(ctypes.byref(p), 1) <= most
    code = ("import ctypes, sys; sys.path[:0] = [%r]\n"
            "from paper_2603_14360_b200 import binding as b\n"
            "f = ctypes.c_void_p(0x10000)\n"
            "for B, T, N in ((2, 144, 84), (2, 512, 84)):\n"      # 9.4 MiB by the plan for speed, at most 8 lean; too much for both
            "    p = b.Params(B=B, T=T, N=N, Nq=N, Nk=N, K=64, V=16, io_dtype=1, gate_kind=1, ckpt_interval=0, dh_clip=0.0)\n"
            "    print(b._lib().m2rnn_bwd_workspace_bytes(ctypes.byref(p), 0) > b.STATIC_SCRATCH_BYTES,\n"
            "          b._lib().m2rnn_bwd_static_scratch(ctypes.byref(p), *([f] * 5), None, None, None, None, None, f, None, *([f] * 5), None, None, None))\n"
            ) % os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}, timeout=300)
    assert r.stdout.split() == ["True", "-6", "True", "-5"], (r.stdout, r.stderr[-2000:])
