"""The binding refuses tensors that a kernel must not be given: on the CPU beside CUDA ones, or laid out in
another order than the kernels read.  Needs no GPU: fake tensors report a CUDA device without one, and
every call below has to be refused before anything is allocated or launched."""
import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

from paper_2603_14360_b200 import binding

B, T, N, V, C = 2, 5, 3, 16, 24


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2603_14360_b200 import build
    build.build()


@pytest.fixture
def fake():
    with FakeTensorMode(allow_non_fake_inputs=True):
        yield lambda *shape, dtype=torch.bfloat16, device="cuda": torch.empty(shape, dtype=dtype, device=device)


def _norm(fake, **over):
    a = dict(y=fake(B, T, N, V), g=fake(B, T, N, V), w=fake(N * V), rstd=fake(B, T, dtype=torch.float32), dout=fake(B, T, N, V))
    return {**a, **over}


def _norm_fwd(a):
    return binding.m2rnn_gated_norm_fwd(a["y"], a["g"], a["w"])


def _norm_bwd(a):
    return binding.m2rnn_gated_norm_bwd(a["y"], a["g"], a["w"], a["rstd"], a["dout"])


NORM = [(_norm_fwd, "y", "y"), (_norm_fwd, "g", "g_in"), (_norm_fwd, "w", "w")]
NORM += [(_norm_bwd, "y", "y"), (_norm_bwd, "g", "g_in"), (_norm_bwd, "w", "w"), (_norm_bwd, "rstd", "rstd"), (_norm_bwd, "dout", "dout")]


@pytest.mark.parametrize("call,arg,name", NORM, ids=lambda x: getattr(x, "__name__", x))
def test_norm_refuses_a_cpu_tensor(fake, call, arg, name):
    good = _norm(fake)
    bad = fake(*good[arg].shape, dtype=good[arg].dtype, device="cpu")
    with pytest.raises(ValueError, match=f"^{name} must be a CUDA tensor"):
        call({**good, arg: bad})


@pytest.mark.parametrize("call,arg,name", [c for c in NORM if c[1] in ("y", "g", "dout")], ids=lambda x: getattr(x, "__name__", x))
@pytest.mark.parametrize("layout", ["permuted", "with gaps"])
def test_norm_refuses_other_layouts(fake, call, arg, name, layout):
    """A dense tensor with two axes exchanged has every element where the kernel looks for another one."""
    bad = fake(B, N, T, V).transpose(1, 2) if layout == "permuted" else fake(B, T, N, 2 * V)[..., :V]
    with pytest.raises(ValueError, match=f"^{name} must be contiguous"):
        call(_norm(fake, **{arg: bad}))


@pytest.mark.parametrize("call", [_norm_fwd, _norm_bwd], ids=lambda f: f.__name__)
def test_norm_refuses_weights_of_another_length(fake, call):
    with pytest.raises(ValueError, match="entries"):
        call(_norm(fake, w=fake(N * V - 8)))


CONV = [(bwd, arg) for bwd in (False, True) for arg in ("x", "w", "bias", "prev")] + [(True, "dout")]


@pytest.mark.parametrize("bwd,arg", CONV)
def test_conv_refuses_a_cpu_tensor(fake, bwd, arg):
    a = dict(x=fake(B, T, C), w=fake(C, 4), bias=fake(C), prev=fake(B, 3, C), dout=fake(B, T, C))
    a[arg] = fake(*a[arg].shape, device="cpu")
    with pytest.raises(ValueError, match=f"^{arg} must be a CUDA tensor"):
        if bwd:
            binding.m2rnn_conv_silu_bwd(a["x"], a["w"], a["dout"], a["bias"], a["prev"])
        else:
            binding.m2rnn_conv_silu_fwd(a["x"], a["w"], a["bias"], a["prev"])


@pytest.mark.parametrize("T,interval,steps", [(256, 0, 200), (200, 8, 192), (9, 2, 8)])
def test_scan_refuses_a_checkpoint_tensor_that_is_too_small(fake, T, interval, steps):
    """The library is not told how long `ckpt` is: 6 sequences of 32 heads, whose checkpoints come every eight steps unless asked otherwise."""
    B, N, K, V, f32 = 6, 32, 64, 16, torch.float32
    q, k, v, W = fake(B, T, 1, K), fake(B, T, 1, K), fake(B, T, N, V), fake(N, V, V)
    out = dict(y=fake(B, T, N, V), hT=fake(B, N, K, V, dtype=f32), ckpt=fake(B, N, steps // (interval or 8), K, V, dtype=f32))
    with pytest.raises(ValueError, match="^ckpt: smaller"):
        binding.m2rnn_fwd(q, k, v, fake(B, T, N, dtype=f32), W, save_ckpt=True, ckpt_interval=interval, out=out)
    out["ckpt"] = fake(B, N, T, K, V, dtype=f32, device="cpu")
    with pytest.raises(ValueError, match="^ckpt must be a CUDA tensor"):
        binding.m2rnn_fwd(q, k, v, fake(B, T, N, dtype=f32), W, save_ckpt=True, ckpt_interval=interval, out=out)
