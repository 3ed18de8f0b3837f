"""Thin binding of ``libm2rnn.so`` (declared in ``include/m2rnn.h``).

Argument marshalling only: every step of the scan runs in the library's CUDA kernels.
torch supplies device memory and the current stream; there is no CPU or eager fallback --
a missing or stale library raises.  The calls of the scan and of the paths around it are marshalled
in C++ (``csrc/py_native.cpp``, built as ``_native.so``): a decoded token takes a few microseconds on
the GPU, so its host path is what counts.  The size queries and self-tests go through ctypes.

    y, hT, ckpt = m2rnn_fwd(q, k, v, gate, W, h0, save_ckpt=True)
    grads       = m2rnn_bwd(q, k, v, gate, W, h0, dy, ckpt=ckpt)
    y1          = m2rnn_decode_step(q1, k1, v1, gate1, W, state)      # state updated in place
    out, rstd   = m2rnn_gated_norm_fwd(y, g_in, w)                    # RMSNorm(y * SiLU(g)) over N*V
    grads       = m2rnn_gated_norm_bwd(y, g_in, w, rstd, dout)        # dy, dg, dw

Tensor layouts are the paper's (Algorithm 1/2): q [B,T,Nq,K], k [B,T,Nk,K], v [B,T,N,V],
gate [B,T,N] fp32, W [N,V,V], h0 [B,N,K,V] fp32.
"""
from __future__ import annotations

import ctypes
import os

import torch

GATE_VALUE, GATE_LOGIT, GATE_PSI = 0, 1, 2
F32, BF16 = 0, 1

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libm2rnn.so")

STATUS = {0: "M2RNN_OK", -1: "M2RNN_ERR_NULL", -2: "M2RNN_ERR_SHAPE", -3: "M2RNN_ERR_UNSUPPORTED",
          -4: "M2RNN_ERR_ALIGN", -5: "M2RNN_ERR_WORKSPACE", -6: "M2RNN_ERR_CUDA", -7: "M2RNN_ERR_TIMEOUT"}


class M2RNNError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        msg = _lib().m2rnn_status_string(status).decode()
        super().__init__(f"{where}: {STATUS.get(status, status)} ({msg})")


class Params(ctypes.Structure):
    """Mirror of ``m2rnn_params``."""
    _fields_ = [("B", ctypes.c_int32), ("T", ctypes.c_int32), ("N", ctypes.c_int32),
                ("Nq", ctypes.c_int32), ("Nk", ctypes.c_int32), ("K", ctypes.c_int32),
                ("V", ctypes.c_int32), ("io_dtype", ctypes.c_int32), ("gate_kind", ctypes.c_int32),
                ("ckpt_interval", ctypes.c_int32), ("dh_clip", ctypes.c_float),
                ("q_stride", ctypes.c_int64), ("k_stride", ctypes.c_int64), ("v_stride", ctypes.c_int64),
                ("total_tokens", ctypes.c_int64), ("cu_seqlens", ctypes.c_void_p)]


_LIB = None
_vp = ctypes.c_void_p
_pp = ctypes.POINTER(Params)

EXPORTS = {
    "m2rnn_version": (ctypes.c_int, []),
    "m2rnn_status_string": (ctypes.c_char_p, [ctypes.c_int]),
    "m2rnn_ckpt_interval": (ctypes.c_int, [_pp]),
    "m2rnn_bwd_row_slab": (ctypes.c_int, [_pp]),
    "m2rnn_ckpt_bytes": (ctypes.c_size_t, [_pp]),
    "m2rnn_fwd_workspace_bytes": (ctypes.c_size_t, [_pp]),
    "m2rnn_fwd": (ctypes.c_int, [_pp] + [_vp] * 13 + [ctypes.c_size_t, _vp, _vp]),
    "m2rnn_bwd_workspace_bytes": (ctypes.c_size_t, [_pp, ctypes.c_int]),
    "m2rnn_bwd": (ctypes.c_int, [_pp] + [_vp] * 19 + [ctypes.c_size_t, _vp, _vp]),
    "m2rnn_bwd_static_scratch": (ctypes.c_int, [_pp] + [_vp] * 20),
    "m2rnn_decode_step": (ctypes.c_int, [_pp] + [_vp] * 12),
    "m2rnn_conv_silu_fwd": (ctypes.c_int, [ctypes.c_int32] * 4 + [_vp, ctypes.c_int64, _vp, _vp, _vp, _vp, ctypes.c_int64, _vp]),
    "m2rnn_conv_silu_bwd_workspace_bytes": (ctypes.c_size_t, [ctypes.c_int32] * 3),
    "m2rnn_conv_silu_bwd": (ctypes.c_int, [ctypes.c_int32] * 4 + [_vp, ctypes.c_int64, _vp, _vp, _vp, _vp, ctypes.c_int64, _vp,
                                             ctypes.c_int64, _vp, _vp, _vp, _vp, ctypes.c_size_t, _vp]),
    "m2rnn_wait_selftest": (ctypes.c_int, [ctypes.c_int64, _vp, _vp, _vp]),
    "m2rnn_gated_norm_fwd": (ctypes.c_int, [ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, _vp, _vp, _vp, ctypes.c_float,
                                            ctypes.c_int32, _vp, _vp, _vp]),
    "m2rnn_gated_norm_bwd_workspace_bytes": (ctypes.c_size_t, [ctypes.c_int64, ctypes.c_int32]),
    "m2rnn_gated_norm_bwd": (ctypes.c_int, [ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, _vp, _vp, _vp, _vp, ctypes.c_int32,
                                            _vp, _vp, _vp, _vp, _vp, ctypes.c_size_t, _vp]),
}

STATIC_SCRATCH_BYTES = 8 << 20   # M2RNN_STATIC_SCRATCH_BYTES


def _lib() -> ctypes.CDLL:
    global _LIB
    if _LIB is None:
        if not os.path.exists(LIB_PATH):
            raise ImportError(f"{LIB_PATH} is not built: run `python -m paper_2603_14360_b200.build` "
                              "(there is no fallback path)")
        lib = ctypes.CDLL(LIB_PATH)
        for name, (res, args) in EXPORTS.items():
            fn = getattr(lib, name)          # AttributeError if the library is stale
            fn.restype, fn.argtypes = res, args
        _LIB = lib
    return _LIB


class _NotLoaded:
    """Stands for the native half until its first use: loads it and takes its own place."""

    def __getattr__(self, name):
        global _native
        _lib()
        from . import _native as mod
        mod.set_error_class(M2RNNError)
        _native = mod
        return getattr(mod, name)


_native = _NotLoaded()


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _stream(stream):
    s = stream if stream is not None else torch.cuda.current_stream()
    return ctypes.c_void_p(s.cuda_stream)


def _io_code(dtype: torch.dtype) -> int:
    if dtype == torch.float32:
        return F32
    if dtype == torch.bfloat16:
        return BF16
    raise TypeError(f"unsupported I/O dtype {dtype}")


def _chk(t, name, shape, dtype, strided_tokens=False):
    if t is None:
        return
    if not t.is_cuda:
        raise ValueError(f"{name} must be a CUDA tensor")
    if tuple(t.shape) != tuple(shape):
        raise ValueError(f"{name}: expected shape {tuple(shape)}, got {tuple(t.shape)}")
    if t.dtype != dtype:
        raise TypeError(f"{name}: expected {dtype}, got {t.dtype}")
    if not t.is_contiguous() and not strided_tokens:     # (q, k, v: _token_stride checks the layout)
        raise ValueError(f"{name} must be contiguous")


def device_status_word(device=None) -> torch.Tensor:
    """The int32 word kernels raise when a bounded wait runs out (one per device, zero = fine)."""
    idx = torch.cuda.current_device() if device is None else torch.device(device).index
    return _native.status_word(idx)


def check_device_status(device=None) -> None:
    """Synchronises and raises if any kernel since the last check reported a timeout."""
    w = device_status_word(device)
    v = int(w.item())
    if v != 0:
        w.zero_()
        raise M2RNNError(v, "device status")


def m2rnn_wait_selftest(limit_cycles: int, device=None, stream=None):
    """Launches the library's wait self-test: one warp waits, with a limit of ``limit_cycles`` SM
    clocks, on a barrier nothing completes.  Returns (status word as the kernel left it, SM clocks
    the wait took); the status must be M2RNN_ERR_TIMEOUT (-7).  Uses words of its own, not the
    device status word of the scan calls."""
    dev = torch.device("cuda", torch.cuda.current_device()) if device is None else torch.device(device)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    waited = torch.zeros(1, dtype=torch.int64, device=dev)
    rc = _lib().m2rnn_wait_selftest(int(limit_cycles), _ptr(status), _ptr(waited), _stream(stream))
    if rc != 0:
        raise M2RNNError(rc, "m2rnn_wait_selftest")
    return int(status.item()), int(waited.item())


def _token_stride(t, name) -> int:
    """Elements between consecutive tokens of q, k or v ([B,T,heads,dim] or packed [tokens,heads,dim]).
    A token's heads must be contiguous and the token axis regular, so that the tensor may be a view
    into a fused projection output; 0 stands for the dense layout."""
    if t.numel() == 0:
        return 0
    if t.stride(-1) != 1 or t.stride(-2) != t.shape[-1]:
        raise ValueError(f"{name}: the heads of a token must be contiguous")
    tok = t.stride(-3)
    if t.dim() == 4 and t.shape[0] > 1 and t.stride(0) != t.shape[1] * tok:
        raise ValueError(f"{name}: batch entries must follow one another along the token axis")
    return 0 if tok == t.shape[-2] * t.shape[-1] else tok


def _params(q, k, v, W, gate_kind, ckpt_interval=0, dh_clip=0.0, decode=False, cu_seqlens=None,
            max_seqlen=None) -> Params:
    if decode:
        B, Nq, K = q.shape
        T, Nk, (N, V) = 1, k.shape[1], v.shape[1:]
        return Params(B, T, N, Nq, Nk, K, V, _io_code(q.dtype), gate_kind, ckpt_interval, dh_clip, 0, 0, 0, 0, None)
    if cu_seqlens is not None:   # packed variable-length batch: q [tokens, Nq, K]
        if cu_seqlens.dtype != torch.int32 or not cu_seqlens.is_cuda or not cu_seqlens.is_contiguous():
            raise TypeError("cu_seqlens must be a contiguous int32 CUDA tensor of B + 1 offsets")
        if max_seqlen is None:
            raise ValueError("max_seqlen (the longest sequence) is required with cu_seqlens")
        total, Nq, K = q.shape
        B, T, Nk, (N, V) = cu_seqlens.numel() - 1, int(max_seqlen), k.shape[1], v.shape[1:]
    else:
        B, T, Nq, K = q.shape
        total, Nk, (N, V) = 0, k.shape[2], v.shape[2:]
    return Params(B, T, N, Nq, Nk, K, V, _io_code(q.dtype), gate_kind, ckpt_interval, dh_clip,
                  _token_stride(q, "q"), _token_stride(k, "k"), _token_stride(v, "v"), total,
                  None if cu_seqlens is None else cu_seqlens.data_ptr())


def m2rnn_version() -> int:
    return _lib().m2rnn_version()


def m2rnn_ckpt_interval(p: Params) -> int:
    c = _lib().m2rnn_ckpt_interval(ctypes.byref(p))
    if c <= 0:
        raise M2RNNError(c, "m2rnn_ckpt_interval")
    return c


def m2rnn_bwd_row_slab(p: Params) -> int:
    r = _lib().m2rnn_bwd_row_slab(ctypes.byref(p))
    if r <= 0:
        raise M2RNNError(r, "m2rnn_bwd_row_slab")
    return r


def m2rnn_bwd_workspace_bytes(p: Params, have_ckpt: bool) -> int:
    return _lib().m2rnn_bwd_workspace_bytes(ctypes.byref(p), int(have_ckpt))


def m2rnn_fwd_workspace_bytes(p: Params) -> int:
    return _lib().m2rnn_fwd_workspace_bytes(ctypes.byref(p))


def m2rnn_fwd(q, k, v, gate, W, h0=None, *, gate_kind=GATE_LOGIT, alpha=None, beta=None, w_r=None,
              save_ckpt=False, ckpt_interval=0, want_hT=True, out=None, workspace=None, stream=None,
              cu_seqlens=None, max_seqlen=None):
    """Forward scan.  Returns (y, hT, ckpt); hT / ckpt are None when not requested.
    ``out`` may hold preallocated ``y`` / ``hT`` / ``ckpt`` tensors to write into; ``workspace``
    a preallocated uint8 tensor of at least ``m2rnn_fwd_workspace_bytes`` bytes (an empty one: do without
    where the library can, at the price of speed).
    q, k, v may be strided views along the token axis (e.g. slices of one fused projection output).
    With ``cu_seqlens`` (int32 [B+1], CUDA) and ``max_seqlen`` the batch is packed: q [tokens,Nq,K],
    k, v, gate [tokens,N], y [tokens,N,V]; states stay [B,N,K,V]."""
    y, hT, ckpt = (out.get("y"), out.get("hT"), out.get("ckpt")) if out else (None, None, None)
    return _native.fwd(q, k, v, gate, W, h0, gate_kind, alpha, beta, w_r, save_ckpt, ckpt_interval, want_hT, y, hT, ckpt,
                       workspace, stream, cu_seqlens, max_seqlen)


def m2rnn_bwd(q, k, v, gate, W, h0, dy, d_hT=None, *, ckpt=None, gate_kind=GATE_LOGIT, alpha=None,
              beta=None, w_r=None, ckpt_interval=0, dh_clip=0.0, want_dh0=True, workspace=None,
              out=None, stream=None, cu_seqlens=None, max_seqlen=None):
    """Backward through time.  Returns dict(dq, dk, dv, dgate, dW, dh0) (dense, whatever the strides
    of q, k, v).  ``cu_seqlens`` / ``max_seqlen``: packed batch, as in ``m2rnn_fwd``."""
    dq, dk, dv, dgate, dW, dh0 = map(out.get, ("dq", "dk", "dv", "dgate", "dW", "dh0")) if out else (None,) * 6
    return _native.bwd(q, k, v, gate, W, h0, dy, d_hT, ckpt, gate_kind, alpha, beta, w_r, ckpt_interval, dh_clip, want_dh0,
                       workspace, dq, dk, dv, dgate, dW, dh0, stream, cu_seqlens, max_seqlen)


def m2rnn_bwd_static_scratch(q, k, v, gate, W, h0, dy, d_hT=None, *, out, ckpt=None, gate_kind=GATE_LOGIT,
                             alpha=None, beta=None, w_r=None, ckpt_interval=0, dh_clip=0.0, stream=None):
    """Backward through time on the library's built-in scratch array, for callers that must not
    allocate device memory (an embedding application that owns the allocator, a service that
    forbids allocation after start-up).  Nothing is allocated here either: ``out`` must already
    hold ``dq, dk, dv, dgate, dW`` (and ``dh0`` if wanted), which are written in place and
    returned.  Problems that need more than ``STATIC_SCRATCH_BYTES`` of scratch raise
    ``M2RNNError`` with ``M2RNN_ERR_WORKSPACE``; calls must not overlap on the GPU, because they
    all share the one array."""
    p = _params(q, k, v, W, gate_kind, ckpt_interval, dh_clip)
    B, T, N, K, V, io = p.B, p.T, p.N, p.K, p.V, q.dtype
    _chk(q, "q", (B, T, p.Nq, K), io); _chk(k, "k", (B, T, p.Nk, K), io); _chk(v, "v", (B, T, N, V), io)
    _chk(gate, "gate", (B, T, N), torch.float32); _chk(W, "W", (N, V, V), io)
    _chk(h0, "h0", (B, N, K, V), torch.float32); _chk(w_r, "w_r", (N, V), io)
    _chk(alpha, "alpha", (N,), torch.float32); _chk(beta, "beta", (N,), torch.float32)
    _chk(dy, "dy", (B, T, N, V), io); _chk(d_hT, "d_hT", (B, N, K, V), torch.float32)
    _chk(out["dq"], "dq", q.shape, io); _chk(out["dk"], "dk", k.shape, io); _chk(out["dv"], "dv", v.shape, io)
    _chk(out["dgate"], "dgate", gate.shape, torch.float32); _chk(out["dW"], "dW", (N, V, V), torch.float32)
    _chk(out.get("dh0"), "dh0", (B, N, K, V), torch.float32)
    rc = _lib().m2rnn_bwd_static_scratch(
        ctypes.byref(p), _ptr(q), _ptr(k), _ptr(v), _ptr(gate), _ptr(W), _ptr(h0), _ptr(alpha), _ptr(beta),
        _ptr(w_r), _ptr(ckpt), _ptr(dy), _ptr(d_hT), _ptr(out["dq"]), _ptr(out["dk"]), _ptr(out["dv"]),
        _ptr(out["dgate"]), _ptr(out["dW"]), _ptr(out.get("dh0")), _ptr(device_status_word(q.device)),
        _stream(stream))
    if rc != 0:
        raise M2RNNError(rc, "m2rnn_bwd_static_scratch")
    return out


def m2rnn_decode_step(q, k, v, gate, W, state, *, gate_kind=GATE_LOGIT, alpha=None, beta=None,
                      w_r=None, y=None, stream=None):
    """One decoding step; ``state`` [B,N,K,V] fp32 is updated in place.  Returns y [B,N,V]."""
    return _native.decode_step(q, k, v, gate, W, state, gate_kind, alpha, beta, w_r, y, stream)


def m2rnn_gated_norm_fwd(y, g_in, w, *, eps=0.0, silu=True, out=None, rstd=None, stream=None):
    """out = RMSNorm(y * SiLU(g_in)) over the head-concatenated features: y, g_in [..., N, V],
    w [N*V] (or [N, V]).  Returns (out like y, rstd [...] fp32)."""
    return _native.gated_norm_fwd(y, g_in, w, eps, silu, out, rstd, stream)


def m2rnn_gated_norm_bwd_workspace_bytes(tokens: int, d: int) -> int:
    return int(_lib().m2rnn_gated_norm_bwd_workspace_bytes(tokens, d))


def m2rnn_gated_norm_bwd(y, g_in, w, rstd, dout, *, silu=True, workspace=None, out=None, stream=None):
    """Backward of m2rnn_gated_norm_fwd -> dict(dy, dg, dw [N*V] fp32)."""
    dy, dg, dw = (out.get("dy"), out.get("dg"), out.get("dw")) if out else (None, None, None)
    return _native.gated_norm_bwd(y, g_in, w, rstd, dout, silu, workspace, dy, dg, dw, stream)


def m2rnn_conv_silu_fwd(x, w, bias=None, prev=None, *, out=None, stream=None):
    """SiLU(depthwise causal conv1d of width 4 along time) of x [B,T,C] (a view into a wider tensor is
    fine); w [C,4], bias [C], prev [B,3,C] (the three inputs before t = 0).  Returns out [B,T,C]."""
    return _native.conv_silu_fwd(x, w, bias, prev, out, stream)


def m2rnn_conv_silu_bwd(x, w, dout, bias=None, prev=None, *, out=None, workspace=None, stream=None):
    """Backward of ``m2rnn_conv_silu_fwd`` -> dict(dx [B,T,C], dw [C,4] fp32, dbias [C] fp32, dprev [B,3,C])."""
    res = dict(out) if out else {}
    res["dx"], res["dw"], res["dbias"], dprev = _native.conv_silu_bwd(
        x, w, dout, bias, prev, workspace, res.get("dx"), res.get("dw"), res.get("dbias"), res.get("dprev"), stream)
    if dprev is not None:
        res["dprev"] = dprev
    return res
