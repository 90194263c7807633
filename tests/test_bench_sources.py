"""The hash by which bench.py tells whether a profile was taken on the current slice-product kernels covers
every local file that those kernels are compiled from."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2503_22875_gb300", "csrc")


def test_kernel_sources_are_the_include_closure():
    todo, seen = ["ozg_gemm.cu", "ozg_gemm_kd.cu"], set()
    while todo:
        f = todo.pop()
        if f not in seen and os.path.exists(os.path.join(CSRC, f)):
            seen.add(f)
            todo += re.findall(r'#include "([^"/]+)"', open(os.path.join(CSRC, f)).read())
    assert set(bench.KERNEL_SOURCES) == seen
