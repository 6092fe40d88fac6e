"""The row-pair kernel's clamp: max(0, M - c) as one half-precision subtraction.

The kernel subtracts whole numbers as half-precision bit patterns (bits v
stand for v * 2^-24) and clamps with .sat, which gives 0 for a negative result
and for a NaN.  numpy's float16 holds the same patterns, so the identity is
checked here over every M the kernel meets, negative ones (two's complement)
included, without a GPU.
"""
import numpy as np
import pytest


def sub_sat(a, b):
    """sub.rn.sat.f16 on bit patterns."""
    x = a.view(np.float16).astype(np.float64) - b.view(np.float16).astype(np.float64)
    x = np.where(np.isnan(x), 0.0, np.clip(x, 0.0, 1.0))
    return x.astype(np.float16).view(np.uint16)


@pytest.mark.parametrize("lo,hi", [(-1023, -1), (0, 382), (383, 2047)])
def test_clamped_subtraction(lo, hi):
    m = np.arange(lo, hi + 1, dtype=np.int64)
    bits = (m & 0xffff).astype(np.uint16)
    for c in [1, 2, 7, 11, 255, 256, 1022, 1023]:
        got = sub_sat(bits, np.full(bits.shape, c, np.uint16)).astype(np.int64)
        np.testing.assert_array_equal(got, np.maximum(0, m - c))
