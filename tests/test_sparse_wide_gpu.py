"""The zero-skipping walk on the GPU at the orders no whole count reaches
(seven and eight row words, and at L(31) counts over 64 bits): plain, hooked
and mirrored parts of a job through the library's launcher, and the batch's
unit function, against the definition summed on the host
(tests/native/sparse_device_check.cu).  Below, counts of the listed orders
with Lemma 2.4's variable held give the whole count's residues."""
import os
import shutil
import subprocess

import pytest

import paper_1507_00315_gb300 as sk
from paper_1507_00315_gb300 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path_factory.mktemp("sparse") / "sparse_device_check")
    subprocess.run([nvcc, "-std=c++17", "-O3", "-maxrregcount=128"] + build.ARCH +
                   ["-cudart", "shared", "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "native", "sparse_device_check.cu"), "-o", exe,
                    build.LIB, "-Xlinker", "-rpath," + build.PKG], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("delta", [0, 1])
@pytest.mark.parametrize("n", range(25, 32))
def test_parts_of_wide_orders(check, delta, n):
    r = subprocess.run([check, str(delta), str(n)], capture_output=True, text=True, timeout=120)
    lines = r.stdout.strip().splitlines()
    assert r.returncode == 0 and lines[-1] == "total bad=0", r.stdout + r.stderr
    assert len(lines) == 1 + 3 + (delta == 0) + (n in (29, 31))


@pytest.mark.parametrize("variant,n", [(0, 13), (0, 16), (1, 15), (2, 14), (2, 15)])
def test_held_variable_gives_the_whole_sum(variant, n):
    whole = sk.count_ex(variant, n, nprimes=4)[1]
    half = sk.count_ex(variant, n, nprimes=4, symmetry=sk.SYMMETRY_NEGATION_EVEN)[1]
    assert half["terms"] == whole["terms"] // 2
    assert half["residues"] == whole["residues"] and any(whole["residues"])
