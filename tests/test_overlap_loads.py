"""Kernels launched with launch overlap read global memory by plain (coherent)
loads only. ld.global.nc (`__ldg`, or what the compiler makes of a
`const __restrict__` parameter) wants memory that nobody writes while the kernel
lives, and a kernel launched with overlap is resident while the one before it
still writes. Read from the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_13660_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    with open(path) as f:
        text = re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _overlaps(text):
    """Whether any launch in a source (or, for a header, in one that includes it) may overlap its predecessor."""
    first = re.findall(r"launch_pdl\(\s*([^,]+?)\s*,", text)
    return any(a != "false" and not a.startswith("bool") for a in first)


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_read_only_loads_where_launches_overlap(path):
    text = _code(path)
    if path.endswith(".cu") and not _overlaps(text):
        return   # plainly launched kernels: everything before them has completed
    assert not re.findall(r"__ldg\b|\bldg[0-9]\b|ld\.global\.nc|ld\.global\.L1::\w+\.nc|__ldlu\b", text)
    assert not re.findall(r"const[^;{}()=]*\*\s*__restrict__", text)


def test_the_rule_sees_both_kinds():
    kinds = {os.path.basename(p): _overlaps(_code(p)) for p in FILES if p.endswith(".cu")}
    assert kinds["block.cu"] is False and not any(kinds[f] is False for f in (
        "accept.cu", "backward.cu", "decode.cu", "forward.cu", "prefill.cu", "xproj.cu"))
