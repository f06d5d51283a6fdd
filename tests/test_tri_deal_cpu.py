"""The rule that sends an SVD block to the reduction with rows in shared memory, for any number of
visible SMs (`tests/tri_deal_host.cu`), and that the eigensolver takes its route from that
rule: a block that no group holds takes the other reduction instead of an error.  No GPU."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.cpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1610_02244_gb300", "csrc")


def test_blocks_are_held_or_take_the_other_route(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "tri_deal_host")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "tri_deal_host.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout


def test_the_eigensolver_routes_by_what_fits():
    with open(os.path.join(CSRC, "heig.cu")) as f:
        src = f.read()
    body = src[src.index("int heig_blocks("):]
    assert body.index("tri_holds(") < body.index("heig_top(")
    assert "<= TRI_ROWS_NMAX)" not in body
