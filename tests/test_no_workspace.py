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
