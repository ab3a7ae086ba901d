"""The hash that ties a committed profile to the kernels covers every header with
device code that btdf_kernels.cu includes."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_1806_09403_gb300", "csrc")


def included(name):
    src = open(os.path.join(CSRC, name)).read()
    return [f for f in re.findall(r'#include "([^"]+)"', src) if os.path.exists(os.path.join(CSRC, f))]


def test_hash_covers_the_device_code_of_the_kernels():
    seen, todo = set(), ["btdf_kernels.cu"]
    while todo:
        f = todo.pop()
        if f not in seen:
            seen.add(f)
            todo += included(f)
    with_code = {f for f in seen if "__device__ __forceinline__" in open(os.path.join(CSRC, f)).read()}
    assert with_code <= set(bench.KERNEL_SOURCES)
