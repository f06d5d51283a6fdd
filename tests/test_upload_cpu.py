"""Host tables on their way to the device: the pinned ring's rules against copies made as late as
they allow (`tests/upload_host.cu`), and that every asynchronous host-to-device copy of the
library goes through it.  No GPU."""
import glob
import os
import re
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.cpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1610_02244_gb300", "csrc")


def test_late_copies_find_their_bytes(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "upload_host")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "upload_host.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout


def test_asynchronous_uploads_go_through_the_ring():
    found = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            src = f.read()
        n = len(re.findall(r"cudaMemcpyAsync\([^;]*cudaMemcpyHostToDevice", src))
        if n:
            found[os.path.basename(path)] = n
    # the ring's own copy, and the one of a table larger than it, which waits for its end
    assert found == {"abi.cu": 2}
