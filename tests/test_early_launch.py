"""Kernels whose launch overlaps the end of the one before (conv, gated norm, decoding step, scans, the sums of partials): a chain in which
each call reads what the one before wrote gives the same bits with the device idle before each call, back to back, behind a copy and
another stream's event, and replayed from a CUDA graph."""
import pytest
import torch

import parity
from paper_2603_14360_b200 import binding, inputs
from paper_2603_14360_b200.inputs import ScanConfig

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,N,V", [(1, 5, 4, 16), (2, 300, 24, 16), (8, 1024, 16, 64)])      # one CTA a kernel; a part wave; many waves
def test_chain_of_dependent_calls(B, T, N, V):
    cfg = ScanConfig("early", B=B, T=T, N=N, K=64, V=V, Nq=1, Nk=1, gate_mean=1.0, w_scale=0.5, seed=3)
    g = parity.to_dev(inputs.make_inputs(cfg))
    C = N * V
    gen = torch.Generator("cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(torch.bfloat16)
    src, w, nw = rnd(B, T, C), rnd(C, 4) * 0.5, rnd(C)
    x, back, state = torch.empty_like(src), torch.empty_like(src), torch.empty_like(g["h0"])
    q, k, gate = g["q"][:, 0].clone(), g["k"][:, 0].clone(), g["gate"][:, 0].clone()

    def chain(stop=lambda: None, move=lambda dst, s: dst.copy_(s)):
        move(x, src)
        move(state, g["h0"])
        res = []
        for _ in range(3):
            stop()
            c = binding.m2rnn_conv_silu_fwd(x, w)
            c = c[0] if isinstance(c, tuple) else c
            stop()
            y, rstd = binding.m2rnn_gated_norm_fwd(c.view(B, T, N, V), src.view(B, T, N, V), nw)
            stop()
            n = binding.m2rnn_gated_norm_bwd(c.view(B, T, N, V), src.view(B, T, N, V), nw, rstd, y)
            stop()
            d = binding.m2rnn_conv_silu_bwd(x, w, n["dy"].reshape(B, T, C).contiguous())
            stop()
            s1 = binding.m2rnn_decode_step(q, k, y[:, -1].contiguous(), gate, g["W"], state)
            stop()
            s2 = binding.m2rnn_decode_step(q, k, s1, gate, g["W"], state)
            stop()
            for to in (torch.bfloat16, torch.float32):
                a = [t.to(to) for t in (g["q"], g["k"], y.view(B, T, N, V))] + [g["gate"], g["W"].to(to), state]
                stop()
                z, hT, ck = binding.m2rnn_fwd(*a, save_ckpt=True)
                stop()
                gr = binding.m2rnn_bwd(*a, z, hT, ckpt=ck)
                stop()
                res += [z, hT, *gr.values()]
            move(x, d["dx"])
            res += [c, y, rstd, *n.values(), *(t for t in d.values() if t is not None), s1, s2]
        stop()
        return res + [state.clone()]

    want = chain(torch.cuda.synchronize)
    same = lambda got: all(torch.equal(a.nan_to_num(), b.nan_to_num()) for a, b in zip(got, want, strict=True))
    assert all(t.float().isfinite().all() for t in want)
    assert same(chain())

    side, other = torch.cuda.Stream(), torch.cuda.Stream()

    def from_other(dst, s):      # written by another stream after this one's reads, waited for through an event
        other.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(other):
            back.view(-1).copy_(src.view(-1))
            dst.copy_(s)
        torch.cuda.current_stream().wait_stream(other)

    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = chain(move=from_other)
    side.synchronize()
    assert same(got)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = chain(move=from_other)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert same(got)
    del graph
