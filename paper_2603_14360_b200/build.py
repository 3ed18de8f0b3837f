"""Builds ``libm2rnn.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU) and the Python
extension ``_native.so`` that calls it with g++ against torch's headers.

    python -m paper_2603_14360_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import concurrent.futures
import importlib.metadata
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libm2rnn.so")
NATIVE = os.path.join(HERE, "_native.so")   # Python extension module: the binding's native half
NATIVE_FOR = os.path.join(OBJ, "native_for.txt")

SOURCES = ["api.cu", "reduce.cu", "scan_f32.cu", "scan_fwd_bf16.cu", "scan_fwd_bf16_cs.cu", "scan_fwd_v16.cu", "scan_fwd_tc.cu", "scan_bwd_bf16.cu", "scan_bwd_v16.cu", "scan_bwd_tc.cu", "decode_bf16.cu", "decode_tc_bf16.cu",
           "bwd_static_scratch.cu", "gated_norm.cu", "conv_silu.cu", "selftest.cu"]

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _newest_header() -> float:
    hdrs = [os.path.join(ROOT, "include", "m2rnn.h")]
    hdrs += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    return max(os.path.getmtime(h) for h in hdrs)


def _compile(src: str, force: bool, verbose: bool) -> str:
    obj = os.path.join(OBJ, src.replace(".cu", ".o"))
    path = os.path.join(CSRC, src)
    if (not force and os.path.exists(obj)
            and os.path.getmtime(obj) >= max(os.path.getmtime(path), _newest_header())):
        return obj
    cmd = ["nvcc", *NVCC_FLAGS, "-c", path, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(f"$ {' '.join(cmd)}\n{r.stdout}{r.stderr}")
    if r.returncode:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def _native_for() -> str:
    """What the extension is built against: it calls into torch's C++ libraries, whose interface is a version's own."""
    return f"torch {importlib.metadata.version('torch')}, Python {sys.version.split()[0]}\n"


def _native_is_current() -> bool:
    src = os.path.join(CSRC, "py_native.cpp")
    newest = max(os.path.getmtime(src), os.path.getmtime(os.path.join(ROOT, "include", "m2rnn.h")))
    if not (os.path.exists(NATIVE) and os.path.getmtime(NATIVE) >= newest and os.path.exists(NATIVE_FOR)):
        return False
    with open(NATIVE_FOR) as f:
        return f.read() == _native_for()


def _build_native(force: bool, verbose: bool) -> None:
    src = os.path.join(CSRC, "py_native.cpp")
    if not force and _native_is_current():
        return
    import sysconfig
    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    inc = [*include_paths("cuda"), sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
    lib = library_paths("cuda")
    tmp = f"{NATIVE}.{os.getpid()}.tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *(f"-I{d}" for d in inc), src, "-o", tmp, f"-L{HERE}", "-l:libm2rnn.so", "-Wl,-rpath,$ORIGIN",
           *(f"-L{d}" for d in lib), "-ltorch_python", "-ltorch", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(f"$ {' '.join(cmd)}\n{r.stdout}{r.stderr}")
    if r.returncode:
        raise RuntimeError("g++ failed on py_native.cpp")
    os.replace(tmp, NATIVE)
    with open(NATIVE_FOR, "w") as f:
        f.write(_native_for())


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    with concurrent.futures.ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
        objs = list(ex.map(lambda s: _compile(s, force, verbose), SOURCES))
    if force or not os.path.exists(LIB) or os.path.getmtime(LIB) < max(os.path.getmtime(o) for o in objs):
        tmp = f"{LIB}.{os.getpid()}.tmp"
        subprocess.check_call(["nvcc", "-shared", "-gencode", "arch=compute_100a,code=sm_100a",
                               "-o", tmp, *objs])
        os.replace(tmp, LIB)
    _build_native(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
