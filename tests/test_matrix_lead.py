"""Which problem of a batch gives the peeling from the matrix its launch shape
(checked on the host; no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_the_largest_matrix_ranked_problem(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = tmp_path / "matrix_lead_check"
    subprocess.check_call([gxx, "-std=c++17", "-O1", os.path.join(HERE, "host", "matrix_lead_check.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and "lead ok" in out.stdout, out.stdout + out.stderr
