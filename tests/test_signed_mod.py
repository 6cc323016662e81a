"""The reduction of an exact item's signed 64-bit sums modulo a prime, on the
host (tests/native/signed_mod_check.cu), against 128-bit arithmetic."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_signed_reduction_over_the_moduli_window(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "signed_mod_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I",
                    os.path.join(ROOT, "paper_1507_00315_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "signed_mod_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.stdout.strip() == "bad=0" and r.returncode == 0
