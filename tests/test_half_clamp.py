"""The row-pair kernels' half-precision arithmetic on whole numbers.

The kernels subtract whole numbers as half-precision bit patterns (bits v
stand for v * 2^-24) and clamp with .sat, which gives 0 for a negative result
and for a NaN; the 16-bit lane also finds the positive halves of a register by
a product with infinity.  numpy's float16 holds the same patterns, so both
identities are checked here over every value the kernels meet, negative ones
(two's complement) included, without a GPU.
"""
import numpy as np
import pytest


def sat(x):
    """The .sat of an exact result: NaN is +0, the rest clamped to [0, 1]."""
    x = np.where(np.isnan(x), 0.0, np.clip(x, 0.0, 1.0))
    return x.astype(np.float16).view(np.uint16)


def sub_sat(a, b):
    """sub.rn.sat.f16 on bit patterns."""
    with np.errstate(invalid="ignore"):
        return sat(a.view(np.float16).astype(np.float64) - b.view(np.float16).astype(np.float64))


@pytest.mark.parametrize("lo,hi", [(-1023, -1), (0, 382), (383, 2047)])
def test_clamped_subtraction(lo, hi):
    """Every opening cost up to the 16-bit lane's clamp (the 8-bit lane's is 1023)."""
    m = np.arange(lo, hi + 1, dtype=np.int64)
    bits = (m & 0xffff).astype(np.uint16)
    for c in range(1, 2048):
        got = sub_sat(bits, np.full(bits.shape, c, np.uint16)).astype(np.int64)
        np.testing.assert_array_equal(got, np.maximum(0, m - c))


def test_positive_halves():
    """x * infinity with .sat: above every score for a positive x, 0 for 0."""
    bits = np.arange(0, 2048, dtype=np.uint16)
    with np.errstate(invalid="ignore"):
        got = sat(bits.view(np.float16).astype(np.float64) * np.inf)
    np.testing.assert_array_equal(got, np.where(bits > 0, 15360, 0))
