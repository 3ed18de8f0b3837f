"""m2rnn_fwd without a workspace: problems that it splits over CTAs for speed only run on whole states."""
import ctypes
import os
import subprocess
import sys

import pytest
import torch

import parity
from paper_2603_14360_b200 import binding, inputs
from paper_2603_14360_b200.inputs import ScanConfig

# B, N, K, V, dtype
OPTIONAL = [(2, 8, 64, 64, "f32"), (1, 3, 16, 16, "f32"), (1, 1, 128, 128, "f32"), (8, 24, 96, 64, "bf16"), (8, 24, 128, 32, "bf16"), (2, 16, 80, 64, "bf16")]
REQUIRED = [(1, 2, 64, 64, "bf16"), (1, 4, 128, 128, "bf16"), (1, 2, 64, 16, "bf16"), (1, 16, 96, 64, "bf16")]   # few units: split to fill the GPU


def _params(case, T=8):
    B, N, K, V, dtype = case
    return binding.Params(B=B, T=T, N=N, Nq=N, Nk=N, K=K, V=V, io_dtype=int(dtype == "bf16"), gate_kind=1, ckpt_interval=0, dh_clip=0.0)


def test_which_problems_need_a_workspace():
    """Where no device is visible an accepted call ends at its launch (-6), a refused one before it (-5)."""
    from paper_2603_14360_b200 import build
    build.build()
    for case in OPTIONAL + REQUIRED:
        assert binding.m2rnn_fwd_workspace_bytes(_params(case)) > 0
    here = os.path.dirname(os.path.abspath(__file__))
    code = ("import ctypes, sys; sys.path[:0] = [%r, %r]\n"
            "import test_no_workspace as t\n"
            "from paper_2603_14360_b200 import binding\n"
            "fake = ctypes.c_void_p(0x10000)\n"
            "for case in t.OPTIONAL + t.REQUIRED:\n"
            "    for ws, n in ((None, 0), (fake, 16)):\n"
            "        print(binding._lib().m2rnn_fwd(ctypes.byref(t._params(case)), *([fake] * 5), None, None, None, None, fake, None, None, ws, n, None, None))\n"
            ) % (here, os.path.dirname(here))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}, timeout=300)
    # a workspace that is too small stays an error
    assert r.stdout.split() == ["-6", "-5"] * len(OPTIONAL) + ["-5", "-5"] * len(REQUIRED), (r.stdout, r.stderr[-2000:])


@pytest.mark.gpu
@pytest.mark.parametrize("case", OPTIONAL, ids=lambda c: "x".join(map(str, c)))
def test_whole_states_without_a_workspace(oracle, case):
    B, N, K, V, dtype = case
    cfg = ScanConfig("nows", B=B, T=21, N=N, K=K, V=V, dtype=dtype, w_scale=0.5, gate_mean=1.0, seed=36)
    d = inputs.make_inputs(cfg, residual=True)
    g = parity.to_dev(d)
    args, kw = [g[x] for x in ("q", "k", "v", "gate", "W", "h0")], dict(w_r=g["w_r"], save_ckpt=True)
    split = binding.m2rnn_fwd(*args, **kw)
    whole = binding.m2rnn_fwd(*args, workspace=torch.empty(0, dtype=torch.uint8, device="cuda"), **kw)
    binding.check_device_status()
    y_ref, hT_ref = parity.oracle_fwd(oracle, cfg, d)
    assert parity.rel_err(whole[0], y_ref) <= parity.TOL[dtype] and parity.rel_err(whole[1], hT_ref) <= parity.TOL[dtype]
    if dtype == "f32":      # the same sums in the same order, however a state is split
        assert all(torch.equal(a, b) for a, b in zip(split, whole))


# B, T, N, K, V, shares of y: where groups of four rows would need more than 4 GiB.  As groups of four while groups of eight would leave
# an SM idle, as groups of eight, on whole states (where those make 16 warps an SM, or eight do not fit either)
LARGE = [(1, 65537, 16, 64, 64, 16), (1, 131072, 16, 64, 64, 16), (4, 32768, 10, 64, 64, 8), (4, 8193, 16, 128, 64, 16), (4, 16384, 16, 128, 64, 16),
         (4, 8192, 16, 128, 128, 16), (4, 16384, 20, 128, 32, 16), (1, 131073, 16, 64, 64, 1), (8, 2049, 64, 64, 64, 1), (8, 2048, 64, 64, 64, 16)]


@pytest.mark.parametrize("case", LARGE, ids=lambda c: "x".join(map(str, c)))
def test_rows_of_large_fp32_problems(case):
    B, T, N, K, V, shares = case
    p = binding.Params(B=B, T=T, N=N, Nq=N, Nk=N, K=K, V=V, io_dtype=0, gate_kind=1, ckpt_interval=0, dh_clip=0.0)
    assert binding.m2rnn_fwd_workspace_bytes(p) == (shares * B * T * N * V * 4 if shares > 1 else 0)


@pytest.mark.gpu
@pytest.mark.parametrize("case", [LARGE[0], LARGE[2], LARGE[5], LARGE[6]], ids=lambda c: "x".join(map(str, c)))
def test_large_fp32_problems_match_whole_states(case):
    """States: bit for bit, however they are split; y too in groups of four rows.  Groups of eight add their two fours first: two orders
    of K / 4 terms each, which differ by at most 2 (K / 4) 2^-24 of the sum of |q_r H_r|, and |H| <= 1 (a mean of tanh and an h0 below 1)."""
    B, T, N, K, V, shares = case
    gen = torch.Generator("cuda").manual_seed(8)
    rnd = lambda *s, std=1.0: torch.empty(s, device="cuda").normal_(0, std, generator=gen)
    q, k, v = rnd(B, T, 1, K, std=K ** -0.5), rnd(B, T, 1, K, std=K ** -0.5), rnd(B, T, N, V)
    args = [q, k, v, rnd(B, T, N) + 1.0, rnd(N, V, V, std=0.5 * V ** -0.5), rnd(B, N, K, V, std=0.1)]
    split = binding.m2rnn_fwd(*args)
    whole = binding.m2rnn_fwd(*args, workspace=torch.empty(0, dtype=torch.uint8, device="cuda"))
    binding.check_device_status()
    assert torch.equal(split[1], whole[1]) and args[5].abs().max() < 1
    if shares == K // 4:
        assert torch.equal(split[0], whole[0])
    else:
        assert ((split[0] - whole[0]).abs().amax(-1) <= K / 2 * 2.0 ** -24 * q.abs().sum(-1)).all()
