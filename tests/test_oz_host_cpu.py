"""The integer pieces of the FP64-accurate GEMM (`csrc/oz.cuh`), compiled for the host
(`tests/oz_host.cu`): the balanced base-128 digits of a value and the rounding of a combined
level sum, against 128-bit integer arithmetic.  No GPU."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.cpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_digits_and_rounding(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "oz_host")
    cmd = [nvcc, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1610_02244_gb300", "csrc"),
           os.path.join(ROOT, "tests", "oz_host.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
    assert "mismatches 0" in r.stdout
