"""A Krylov step's result slot (`csrc/krylov_slot.cuh`): the status word is read with every step,
and an expired device-side wait is an error however finite the step's numbers are.  No GPU."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.cpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1610_02244_gb300", "csrc")


def test_expired_wait_is_reported_with_finite_numbers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "krylov_slot_host")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "krylov_slot_host.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout


def test_every_step_is_judged_by_its_slot():
    with open(os.path.join(CSRC, "lanczos.cu")) as f:
        src = f.read()
    step = src[src.index("auto check_step"):]
    step = step[:step.index("\n  };")]
    assert "slot_state(" in step and "SLOT_TIMEOUT" in step
