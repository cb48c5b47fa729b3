"""The 32-bit layout arithmetic of the kernels against the 64-bit one, which
test_layout_cpu.py pins, compiled from the library's header and run on the
host."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_layout_arithmetic_32():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "layout32_check")
        subprocess.run([nvcc, "-std=c++17", "-O1", os.path.join(HERE, "layout32_check.cu"), "-o", exe],
                       check=True, capture_output=True)
        r = subprocess.run([exe], capture_output=True, text=True)
        assert r.stdout.strip() == "ok" and r.returncode == 0, r.stdout + r.stderr
