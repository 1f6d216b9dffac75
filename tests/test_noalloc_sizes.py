"""The allocation-free selection takes every size it took when it was
introduced (checked on the host; no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_sizes_of_the_first_range_still_fit(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = tmp_path / "noalloc_check"
    subprocess.check_call([gxx, "-std=c++17", "-O1", os.path.join(HERE, "host", "noalloc_check.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    assert "noalloc ok" in out.stdout
