"""The pool of streams and memory behind the synchronous calls, on the host
against a fake CUDA runtime (tests/native/call_pool_check.cpp): a set goes back
only when nothing of the call is in flight, on error paths too."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sets_go_back_drained(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "call_pool_check")
    csrc = os.path.join(ROOT, "paper_1507_00315_gb300", "csrc")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-cudart", "shared", "-I", csrc,
                    os.path.join(csrc, "sk_pool.cu"),
                    os.path.join(ROOT, "tests", "native", "call_pool_check.cpp"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    lines = r.stdout.strip().splitlines()
    assert lines[-1] == "total bad=0" and r.returncode == 0, r.stdout
