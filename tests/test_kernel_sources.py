"""The kernels are launched programmatically: their blocks wait while the kernel before still writes.  So nothing that a
kernel reads is read-only for its whole life, and no source may take the read-only path (CPU: reads the sources)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_14530_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_loads(path):
    code = _code(path)
    assert not re.search(r"__ldg\w*\s*\(|ld\.global\.nc", code)
    assert not re.search(r"const\s+\w+\s*\*\s*(const\s+)?__restrict__", code)


def test_kernels_wait_before_they_read():
    """Every kernel calls pdl_entry."""
    for path in SOURCES:
        code = _code(path)
        for m in re.finditer(r"__global__", code):
            nxt = code.find("__global__", m.end())
            assert "pdl_entry(" in code[m.start():nxt if nxt >= 0 else len(code)], (path, code[m.start():m.start() + 120])
