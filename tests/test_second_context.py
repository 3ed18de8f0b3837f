"""The library in two contexts of one device, one after the other (its own process): kernel limits and
addresses that belong to a context are asked for again in the next."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r"""
import ctypes, sys
sys.path.insert(0, %r)
from paper_2603_14360_b200.binding import EXPORTS, LIB_PATH, Params
cu = ctypes.CDLL("libcuda.so.1")
lib = ctypes.CDLL(LIB_PATH)
for name, (res, args) in EXPORTS.items():
    getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
vp, sz = ctypes.c_void_p, ctypes.c_size_t

def buf(n):      # n zero bytes on the device
    p = vp()
    assert cu.cuMemAlloc_v2(ctypes.byref(p), sz(n)) == 0 and cu.cuMemsetD8_v2(p, 0, sz(n)) == 0
    return p

def run():
    B, T, N, K, V = 1, 40, 200, 64, 64      # a state to a CTA: more shared memory than a kernel has unasked
    p = Params(B, T, N, N, N, K, V, 1, 1, 0, 0.0)
    vec, gate, W, state = buf(2 * T * N * K), buf(4 * T * N), buf(2 * N * V * V), buf(4 * N * K * V)
    y, status = buf(2 * T * N * V), buf(4)
    assert lib.m2rnn_fwd_workspace_bytes(ctypes.byref(p)) == 0
    rc = [lib.m2rnn_fwd(ctypes.byref(p), vec, vec, vec, gate, W, None, None, None, None, y, state, None, None, 0, status, None)]
    p = Params(B, 20, 2, 2, 2, 16, 16, 0, 1, 0, 0.0)
    out = [buf(4 * 20 * 2 * 16) for _ in range(3)] + [buf(4 * 20 * 2), buf(4 * 2 * 256)]
    rc.append(lib.m2rnn_bwd_static_scratch(ctypes.byref(p), vec, vec, vec, gate, W, None, None, None, None, None, vec, None, *out, None, status, None))
    rc.append(cu.cuCtxSynchronize())
    word = ctypes.c_int(1)
    assert cu.cuMemcpyDtoH_v2(ctypes.byref(word), status, sz(4)) == 0
    return rc + [word.value]

assert cu.cuInit(0) == 0
for _ in range(2):
    ctx = vp()
    assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0) == 0      # current from here on
    print(run())
"""


@pytest.mark.gpu
def test_scans_in_a_second_context():
    r = subprocess.run([sys.executable, "-c", CODE % ROOT], capture_output=True, text=True, timeout=300)
    assert r.stdout.split("\n")[:2] == ["[0, 0, 0, 0]"] * 2, (r.stdout, r.stderr[-2000:])
