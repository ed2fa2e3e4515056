"""The library's kernels overlap along a stream: a kernel is resident while
the one before it still writes.  The read-only load path (ld.global.nc, by
__ldg or chosen by the compiler for `const __restrict__` pointers) is defined
only for memory that nobody writes while the kernel is resident, so the sources
may use it for the caller's K and V rows and for nothing else."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2606_14782_gb300", "csrc")
SOURCES = sorted(p for ext in ("cu", "cuh", "h") for p in glob.glob(os.path.join(CSRC, "*." + ext)))


def _code(path):
    with open(path) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_only_caller_rows_take_the_read_only_path(path):
    code = _code(path)
    for word in ("__restrict", "ld.global.nc"):
        assert word not in code, word
    helper = 1 if os.path.basename(path) == "common.cuh" else 0
    assert len(re.findall(r"\b__ldg\b", code)) == helper  # inside load_input
    calls = re.findall(r"= load_input\(([^;]*)\);", code)
    assert all(re.match(r"tab\.[kv]\[", c) for c in calls), calls


def test_the_sources_are_found():
    names = {os.path.basename(p) for p in SOURCES}
    assert {"common.cuh", "calibrate.cu", "select.cuh", "window_tc.cu"} <= names
    assert sum(len(re.findall(r"\bload_input\(tab", _code(p))) for p in SOURCES) == 4
