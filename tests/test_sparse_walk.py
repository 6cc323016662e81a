"""The zero-skipping walk's tables, tile set-up and products on the host, for
every (delta, n) the library compiles (tests/native/sparse_walk_check.cu):
addresses inside the tables, factors and zero masks equal to the definition,
products exact, every assignment covered once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_walk_on_the_host(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "sparse_walk_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I",
                    os.path.join(ROOT, "paper_1507_00315_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "sparse_walk_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    lines = r.stdout.strip().splitlines()
    assert lines[-1] == "total bad=0", "\n".join(l for l in lines if not l.endswith("bad=0"))
    assert r.returncode == 0
    assert len(lines) == 2 * 19 + 5 + 2 + 1
