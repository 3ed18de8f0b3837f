"""Raising a kernel's limit of shared memory, with threads and contexts that get in each other's way: the
bookkeeping is plain C++ and runs here against a stand-in for the runtime (no GPU)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2603_14360_b200", "csrc")


def test_limits_hold_for_every_thread_and_context(tmp_path):
    exe = str(tmp_path / "smem_limit_test")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-Wall", "-Werror", "-I", CSRC, os.path.join(HERE, "smem_limit_test.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
