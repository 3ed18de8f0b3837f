"""The input path before the scan (SiLU of a depthwise causal conv1d of width 4 over the q, k, v
projections) against the fp64 oracle, forward and backward; and the chain conv -> strided views ->
scan that the library is meant to be used in."""
import pytest
import torch

import parity
from paper_2603_14360_b200 import binding, inputs
from paper_2603_14360_b200.inputs import ScanConfig

pytestmark = pytest.mark.gpu
F = inputs.to_f64

SHAPES = [(2, 37, 64), (1, 1, 8), (3, 200, 328), (1, 64, 8), (2, 129, 1032), (4, 3, 16)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("with_prev", [False, True])
def test_forward_backward(oracle, dtype, shape, with_prev):
    B, T, C = shape
    d = inputs.make_conv_inputs(B, T, C, dtype, seed=500 + T, prev=with_prev)
    g = {k: (None if v is None else v.cuda()) for k, v in d.items()}
    tol = parity.TOL[dtype]
    out = binding.m2rnn_conv_silu_fwd(g["x"], g["w"], g["bias"], g["prev"])
    ref = oracle.conv_silu_fwd(F(d["x"]), F(d["w"]), F(d["bias"]), F(d["prev"]))
    assert parity.rel_err(out, ref) <= tol
    got = binding.m2rnn_conv_silu_bwd(g["x"], g["w"], g["dout"], g["bias"], g["prev"])
    want = oracle.conv_silu_bwd(F(d["x"]), F(d["w"]), F(d["dout"]), F(d["bias"]), F(d["prev"]))
    for name in ("dx", "dw", "dbias") + (("dprev",) if with_prev else ()):
        assert parity.rel_err(got[name], want[name]) <= tol, name
    again = binding.m2rnn_conv_silu_bwd(g["x"], g["w"], g["dout"], g["bias"], g["prev"])
    assert all(torch.equal(again[x], got[x]) for x in got if got[x] is not None)     # fixed-order sums


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(9, 130, 520), (10, 193, 1032), (33, 1, 1032), (34, 257, 1032)], ids=lambda s: "x".join(map(str, s)))
def test_steps_per_thread(oracle, dtype, shape):
    """Problems on both sides of the lines between 16, 32 and 64 time steps per thread, with a ragged last tile."""
    test_forward_backward(oracle, dtype, shape, True)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_runs_that_make_rounds_come_out_even(oracle, dtype):
    """Enough for runs of 64 steps: the backward's runs are of other lengths, neither a multiple of a batch nor of the sequence."""
    test_forward_backward(oracle, dtype, (3, 2101, 1608), True)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_large_inputs(oracle, dtype):
    """SiLU and its derivative far out, where the sigmoid is 0 or 1: one tap, so that the products are exact in either type."""
    d = inputs.make_conv_inputs(2, 40, 64, dtype, seed=17, prev=False)
    d["w"].zero_(); d["w"][:, 3] = 1.0
    d["bias"].zero_()
    d["x"] = (d["x"].float() * 2.0 ** torch.arange(40).sub(10)[None, :, None]).to(d["x"].dtype)
    g = {k: (None if v is None else v.cuda()) for k, v in d.items()}
    out, ref = binding.m2rnn_conv_silu_fwd(g["x"], g["w"], g["bias"]), oracle.conv_silu_fwd(F(d["x"]), F(d["w"]), F(d["bias"]))
    got = binding.m2rnn_conv_silu_bwd(g["x"], g["w"], g["dout"], g["bias"])
    want = oracle.conv_silu_bwd(F(d["x"]), F(d["w"]), F(d["dout"]), F(d["bias"]))
    for t in range(40):       # by itself: a large step would hide the others
        assert parity.rel_err(out[:, t], ref[:, t]) <= parity.TOL[dtype] and parity.rel_err(got["dx"][:, t], want["dx"][:, t]) <= parity.TOL[dtype], t


def test_no_bias_and_empty(oracle):
    d = inputs.make_conv_inputs(2, 19, 32, "f32", seed=9, prev=False)
    g = {k: (None if v is None else v.cuda()) for k, v in d.items()}
    out = binding.m2rnn_conv_silu_fwd(g["x"], g["w"])
    assert parity.rel_err(out, oracle.conv_silu_fwd(F(d["x"]), F(d["w"]))) <= 1e-4
    e = binding.m2rnn_conv_silu_fwd(g["x"][:, :0], g["w"])
    assert e.shape == (2, 0, 32)
    r = binding.m2rnn_conv_silu_bwd(g["x"][:, :0].contiguous(), g["w"], g["dout"][:, :0].contiguous())
    assert float(r["dw"].abs().max()) == 0.0


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_fused_projection_through_conv_into_the_scan(oracle, dtype):
    """One [B,T,Nq K + Nk K + N V] projection tensor -> one conv call in place of three -> column
    slices of its output as the scan's strided q, k, v; backward the same way round."""
    cfg = ScanConfig("chain", B=2, T=45, N=4, K=32, V=16, Nq=1, Nk=1, dtype=dtype, gate_mean=1.0, seed=91)
    wq, wv = cfg.nq * cfg.K, cfg.N * cfg.V
    C = 2 * wq + wv
    d = inputs.make_conv_inputs(cfg.B, cfg.T, C, dtype, seed=92, prev=False)
    s = inputs.make_inputs(cfg, backward=True)
    g = {k: (None if v is None else v.cuda()) for k, v in d.items()}
    gs = parity.to_dev(s)
    act = binding.m2rnn_conv_silu_fwd(g["x"], g["w"], g["bias"])
    q = act[..., :wq].unflatten(2, (cfg.nq, cfg.K))
    k = act[..., wq:2 * wq].unflatten(2, (cfg.nk, cfg.K))
    v = act[..., 2 * wq:].unflatten(2, (cfg.N, cfg.V))
    y, hT, ckpt = binding.m2rnn_fwd(q, k, v, gs["gate"], gs["W"], gs["h0"], save_ckpt=True)
    grads = binding.m2rnn_bwd(q, k, v, gs["gate"], gs["W"], gs["h0"], gs["dy"], ckpt=ckpt)
    dact = torch.cat([grads["dq"].flatten(2), grads["dk"].flatten(2), grads["dv"].flatten(2)], dim=2)
    back = binding.m2rnn_conv_silu_bwd(g["x"], g["w"], dact, g["bias"])
    binding.check_device_status()
    # the oracle, step by step in fp64 from the same inputs
    act_ref = oracle.conv_silu_fwd(F(d["x"]), F(d["w"]), F(d["bias"]))
    qr, kr = act_ref[..., :wq].reshape(cfg.B, cfg.T, cfg.nq, cfg.K), act_ref[..., wq:2 * wq].reshape(cfg.B, cfg.T, cfg.nk, cfg.K)
    vr = act_ref[..., 2 * wq:].reshape(cfg.B, cfg.T, cfg.N, cfg.V)
    y_ref, hT_ref = oracle.fwd(qr, kr, vr, F(s["gate"]), F(s["W"]), F(s["h0"]))
    r = oracle.bwd(qr, kr, vr, F(s["gate"]), F(s["W"]), F(s["h0"]), F(s["dy"]))
    import numpy as np
    dact_ref = np.concatenate([r["dq"].reshape(cfg.B, cfg.T, -1), r["dk"].reshape(cfg.B, cfg.T, -1), r["dv"].reshape(cfg.B, cfg.T, -1)], axis=2)
    back_ref = oracle.conv_silu_bwd(F(d["x"]), F(d["w"]), dact_ref, F(d["bias"]))
    tol = parity.TOL[dtype]
    assert parity.rel_err(y, y_ref) <= tol and parity.rel_err(hT, hT_ref) <= tol
    for name in ("dx", "dw", "dbias"):
        assert parity.rel_err(back[name], back_ref[name]) <= tol, name


@pytest.mark.parametrize("with_prev", [False, True])
def test_fp32_sigmoid_over_its_whole_range(with_prev):
    """fp32, pre-activations from -100 to 100 and both zeros, element by element: out = pre s(pre) and dx = dout SiLU'(pre).

    Taps (0, 0, 0, 1) make pre = x and dx = dpre.  The sigmoid is r or e r with e = exp(-|x|), r = 1/(1 + e): expf is good to
    2 ulp, a Newton step leaves r within 2, and the product, the sum 1 + e and out are rounded: 8 ulp = 2^-20 relative,
    wherever the result is a normal number (below, its spacing 2^-149).  SiLU' = s (1 + x (1 - s)) cancels near its zero at
    -1.278 and where 1 - s does, so its error is against s (1 + |x| (1 - s)), with 1 - s good to 2^-24 absolute."""
    x = torch.cat([torch.linspace(-100, 100, 2001), torch.tensor([0.0, -0.0, 1e-30, -1e-30, 87.0, -87.0, 88.5, -88.5, -88.8]),
                   torch.linspace(-1.3, -1.25, 38)])
    T = x.numel() // 4
    x = x[:4 * T].reshape(1, T, 4).contiguous()
    w = torch.tensor([[0.0, 0.0, 0.0, 1.0]]).repeat(4, 1)
    dout = torch.full_like(x, 1.0)
    prev = torch.zeros(1, 3, 4).cuda() if with_prev else None
    out = binding.m2rnn_conv_silu_fwd(x.cuda(), w.cuda(), None, prev).cpu().double()
    dx = binding.m2rnn_conv_silu_bwd(x.cuda(), w.cuda(), dout.cuda(), None, prev)["dx"].cpu().double()
    z = x.double()
    s, t = torch.sigmoid(z), torch.sigmoid(-z)
    assert ((out - z * s).abs() <= 2.0 ** -20 * (z * s).abs() + 2.0 ** -148 * (1 + z.abs())).all()
    bound = 2.0 ** -20 * s * (1 + z.abs() * t) + 2.0 ** -24 * s * z.abs() + 2.0 ** -148 * (1 + z.abs())
    assert ((dx - s * (1 + z * t)).abs() <= bound).all()
