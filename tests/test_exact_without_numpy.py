"""The exact calls' argument and result conversion needs nothing but the
standard library: the words of a result array as rows of Python integers, in
a process where numpy cannot be imported."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rows_of_a_result():
    code = ("import sys, ctypes; sys.modules['numpy'] = None\n"
            "import paper_1507_00315_gb300 as sk\n"
            "v = [2**64 - 1 - 3 * i for i in range(24)]\n"
            "for k in (1, 3, 4):\n"
            "    got = sk._rows((ctypes.c_uint64 * 24)(*v), k)\n"
            "    assert got == [v[i:i + k] for i in range(0, 24, k)]\n"
            "    assert all(type(x) is int for r in got for x in r)\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
