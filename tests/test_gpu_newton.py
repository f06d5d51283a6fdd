"""`rsqrt_newton` and `rcp_newton` (csrc/f32conv.cuh), which the reflectors, the pivots of the inverse
iteration, the Krylov norms and the SVD's selection use, over their mantissas, exponents and
signs (`tests/newton_gpu.cu`).  Bounds, derived beside the functions: one rounding (2^-53) for the
reciprocal, one and a half for the reciprocal root; 0.001 of one for terms of order 2^-60."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_newton_steps(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "newton")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                        "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "paper_1610_02244_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "newton_gpu.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
