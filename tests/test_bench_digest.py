"""The source digest that decides whether stored ncu counters still describe a
kernel (CPU): a change in any part of the kernel changes it."""
import os

import pytest

import bench

SRC = os.path.join(os.path.dirname(bench.__file__), "paper_1605_01522_gb300", "csrc", "kernels.cu")


@pytest.mark.parametrize("kernel,part,old", [
    ("spmv_warp<3x3,f64>", "struct KSpmvWarp", "a.alpha * s"),
    ("smooth_warp<3x3,f32>", "struct KSmoothWarp", "xi + dd"),
    ("smooth_warp<3x3,f32>", "bsr_row(", "acc[r] += "),
    ("smooth_sell4<3x3,f32>", "struct KSmoothSell ", "d_smooth"),
    ("smooth_sell_split<3x3,f32>", "struct KSmoothSellSplit", "a.x[i] + dd"),
    ("spmv_sell_split<1x1,f32>", "sell_split_entry(", "part[h]"),
    ("spmv_rows<5x5,f64>", "struct KSpmvRows", "bid - a.end"),
])
def test_digest_covers_every_part_of_a_kernel(kernel, part, old):
    src = open(SRC).read()
    d = bench.kernel_source_digest(kernel)
    assert d and d == bench.kernel_source_digest(kernel, src)
    at = src.index(old, src.index(part))
    assert d != bench.kernel_source_digest(kernel, src[:at] + "/**/" + src[at:])
    assert d == bench.kernel_source_digest(kernel, src + "// elsewhere")
