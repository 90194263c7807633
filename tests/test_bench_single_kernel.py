"""The kernel and product count that bench.py's single-call roofline names are those of the call's plan."""
import pytest

import bench
from paper_2503_22875_gb300 import build, ozg


@pytest.mark.parametrize("n,s,kernel,products", [
    (8192, 7, "kd", 19), (4096, 10, "kd", 35), (4096, 11, "stacked", 66), (8192, 12, "stacked", 78),
    (32768, 7, "stacked", 28), (1024, 8, "split", 36), (4096, 18, "", 171)])
def test_kernel_of_a_single_call(n, s, kernel, products):
    build.build()
    name, count, variant = bench.single_kernel(ozg, 152, n, s)
    assert (name, count) == (f"slice_gemm_{kernel}_kernel".replace("__", "_"), products)
    assert variant == (5 if kernel in ("stacked", "split") else None)


def test_a_profile_is_that_of_the_kernel():
    kernels = [f"slice_gemm_{x}_kernel" for x in ("kd", "split", "stacked")]
    names = [bench.single_profile(x, 8192, 7) for x in kernels]
    assert names == ["slice_gemm_kd_8192_s7", "slice_gemm_split_8192_s7", "slice_gemm_8192_s7"]
    assert bench.profile_traffic(names[2])[2] == 5  # tile variant 5: the stacked kernel
