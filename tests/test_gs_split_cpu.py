"""Where the one-launch Gram-Schmidt step applies, for any number of visible SMs
(`tests/gs_split_host.cu`); elsewhere the separate launches do the step.  No GPU."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.cpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1610_02244_gb300", "csrc")


def test_slices_fit_where_the_step_applies(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "gs_split_host")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "gs_split_host.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout


def test_the_solver_asks_what_fits_its_device():
    with open(os.path.join(CSRC, "kernels_f64.cu")) as f:
        src = f.read()
    assert "vec_gs_eligible(const Ctx* c, int64_t n) { return gs_fits(n, c->nsm); }" in src
