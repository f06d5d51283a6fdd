"""Device properties and kernel attributes belong to a context's device: no translation unit keeps
them behind a static of a function, which would hold for the first device of the process only.
No GPU."""
import glob
import os
import re

import pytest

pytestmark = pytest.mark.cpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_02244_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), f.read()


def test_shared_memory_limits_are_raised_per_context():
    where = {name: src.count("cudaFuncSetAttribute(") for name, src in sources() if "cudaFuncSetAttribute(" in src}
    assert where == {"abi.cu": 1}  # func_smem


def test_no_function_static_holds_a_device_property():
    for name, src in sources():
        for m in re.finditer(r"^[ \t]+static (?:int|size_t|bool) \w+(?: = \w+)?(?:, \w+ = \w+)*;", src, re.M):
            raise AssertionError(f"{name}: {m.group(0).strip()}")
