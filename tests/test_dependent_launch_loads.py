"""Kernels that are launched as programmatic dependents are alive while the previous kernel still writes what they will
read.  The read-only (non-coherent) load path requires data that nothing writes during the kernel, so no source
that such a kernel is built from uses it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1302_2132_gb300", "csrc")


def test_no_read_only_loads():
    files = {os.path.basename(f): open(f).read() for f in glob.glob(os.path.join(CSRC, "*.cu*"))}
    waiting = {f for f, s in files.items() if "griddepcontrol.wait" in s}
    assert {"gks_step.cuh", "gks_curv_step.cuh"} <= waiting
    reached = set()

    def reach(f):
        if f in files and f not in reached:
            reached.add(f)
            for g in re.findall(r'#include "([^"]+)"', files[f]):
                reach(g)

    for f in waiting:
        reach(f)
    for f in reached:
        code = re.sub(r"//[^\n]*", "", files[f])
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc|__restrict__", code), f
