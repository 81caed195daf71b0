"""The integer doubling of the FP64 passes (dq_math.cuh, twice) against x + x, by its
formula, over every exponent: zeros, subnormals (whose carry enters the exponent),
normals, the two largest exponents (overflow), infinities.  No GPU."""
import numpy as np
import pytest


def twice_bits(b):
    hi, lo = (b >> np.uint64(32)).astype(np.uint32), b.astype(np.uint32)
    e, sign = hi & np.uint32(0x7ff00000), hi & np.uint32(0x80000000)
    up = (hi << np.uint32(1)) | (lo >> np.uint32(31))
    h = np.where(e != 0, hi + np.uint32(0x00100000), sign | (up & np.uint32(0x7fffffff)))
    low = np.where(e != 0, lo, lo << np.uint32(1))
    top, inf = e >= np.uint32(0x7fe00000), e == np.uint32(0x7ff00000)
    h = np.where(top, np.where(inf, hi, sign | np.uint32(0x7ff00000)), h)
    low = np.where(top, np.where(inf, lo, np.uint32(0)), low)
    return (h.astype(np.uint64) << np.uint64(32)) | low.astype(np.uint64)


@pytest.mark.parametrize("mantissa", ["edges", "random"])
def test_twice_is_x_plus_x(mantissa):
    if mantissa == "edges":
        m = np.array([0, 1, 2, 0x80000000, 0xffffffff, 1 << 32, (1 << 51) - 1, 1 << 51, (1 << 52) - 1], dtype=np.uint64)
    else:
        m = np.random.default_rng(0).integers(0, 1 << 52, 200, dtype=np.uint64)
    b = ((np.arange(4096, dtype=np.uint64) << np.uint64(52))[:, None] | m[None]).ravel()
    x = b.view(np.float64)
    with np.errstate(all="ignore"):
        want = x + x
    got = twice_bits(b).view(np.float64)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
