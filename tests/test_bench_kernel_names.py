"""bench.py's roofline entry names kernels that exist, and for the prefill the
one that its workspace selects."""
import glob
import os
import re

import bench


def test_kernel_names_are_those_of_the_sources():
    csrc = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2401_13660_gb300", "csrc", "*.cu")
    text = "".join(open(f).read() for f in glob.glob(csrc))
    kernels = set(re.findall(r"__global__[^;{]*?(\w+_kernel)\s*\(", text))
    for group in ("prefill", "verify", "rollback", "step"):
        for ws in (256, 1 << 20):
            assert bench.kernel_name(group, ws) in kernels
    assert bench.kernel_name("prefill", 256) != bench.kernel_name("prefill", 1 << 20)
