"""The bulk prefetches into L2 name their elements, and prefetch_l2 alone turns
a count into bytes: a count times a fixed width reached past the end of the
32-bit depth keys (CPU; reads the sources)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_16298_gb300", "csrc")


def test_prefetches_count_elements():
    calls = []
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        code = re.sub(r"template <typename T>\s*__device__ __forceinline__ void prefetch_l2\(const T\* p, uint32_t n\)",
                      "", code)
        calls += re.findall(r"prefetch_l2\(([^;]*)\);", code)
    assert len(calls) >= 7
    for c in calls:
        assert "*" not in c and "sizeof" not in c, c
