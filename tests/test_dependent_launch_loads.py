"""Kernels under programmatic dependent launch are resident while the launch
before them may still write: their sources have no read-only loads (__ldg, or
a const __restrict__ pointer), whose contract is data that nobody writes as
long as the kernel runs (CPU; reads the sources)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_16298_gb300", "csrc")
# every source with such a kernel, and the headers they share
SOURCES = sorted(f for f in glob.glob(os.path.join(CSRC, "*.cu*")) if "begin_launch()" in open(f).read()
                 or os.path.basename(f) in ("onesweep.cuh", "project.cuh", "render.cuh"))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_loads(path):
    code = re.sub(r"//[^\n]*", "", open(path).read())
    assert "__ldg(" not in code
    assert not re.findall(r"const\s+[\w:<>]+\s*\*\s*(?:const\s*\*?\s*)?__restrict__", code)


def test_every_dependent_launch_waits():
    """launch_after only takes kernels that start with begin_launch()."""
    for path in SOURCES:
        code = re.sub(r"//[^\n]*", "", open(path).read())
        kernels = re.split(r"__global__", code)[1:]
        waits = {re.search(r"\b(k_\w+)\s*\(", k).group(1): "begin_launch();" in k for k in kernels}
        for name in re.findall(r"launch_after\((?:\w+::)?(k_\w+)", code):
            assert waits[name], name


def test_depth_sort_reads_its_own_launch_coherently():
    """The single-launch depth sort writes counts and values that other blocks
    of the launch read: only the records, which it never writes, may take the
    read-only path, and the bulk copy of the values follows a proxy fence over
    global memory too."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "depth_sort.cu")).read())
    assert re.findall(r"__ldg\((\w+)", code) == ["s_g"]
    copy = code.index("bulk_g2s(")
    assert code.rindex("fence.proxy.async;", 0, copy) > code.rindex("mbar_init(", 0, copy)
