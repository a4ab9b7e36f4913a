"""Kernels launched with programmatic stream serialisation are resident before the kernel ahead of them has
finished, so the arrays they read are not constant over their lifetime, which read-only (non-coherent) loads ask for:
the library's sources use none, and no pointer is declared free of aliases (which lets the compiler use them)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_17950_gb300", "csrc")


def test_no_read_only_loads_of_arrays_that_kernels_write():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert len(files) >= 9
    for f in files:
        code = re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", open(f).read()), flags=re.S)
        found = re.findall(r"__ldg\s*\(|__restrict__|ld\.global(?:\.\w+)*\.nc|tex1Dfetch", code)
        assert not found, (os.path.basename(f), found)
