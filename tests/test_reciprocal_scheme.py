"""The kernels' reciprocal (Newton's iteration from the single-precision reciprocal of the
significand, exponents moved by integer operations), restated on the CPU with exact fused
operations: within 1.5 units in the last place over its range of exponents."""
import struct
from fractions import Fraction

import numpy as np
import pytest


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))  # one rounding, to nearest even


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _recip(x):
    b = _bits(x)
    hi, lo = b >> 32, b & 0xffffffff
    ex = (hi >> 20) & 0x7ff
    assert 2 <= ex <= 2044
    fm = np.array([0x3f800000 | ((hi & 0xfffff) << 3) | (lo >> 29)], np.uint32).view(np.float32)
    fr = int((np.float32(1.0) / fm).view(np.uint32)[0])
    fe = (fr >> 23) - 127
    rh = (hi & 0x80000000) | ((1023 + fe + 1023 - ex) << 20) | ((fr & 0x7fffff) >> 3)
    r = struct.unpack("<d", struct.pack("<Q", (rh << 32) | ((fr << 29) & 0xffffffff)))[0]
    for _ in range(2):
        r = _fma(r, _fma(-x, r, 1.0), r)
    return r


@pytest.mark.parametrize("e", [-1021, -1020, -300, -1, 0, 1, 52, 1000, 1020, 1021])
def test_reciprocal_within_one_and_a_half_units(e):
    rng = np.random.default_rng(e + 2000)
    sig = [1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -23, 1.5] + list(rng.uniform(1.0, 2.0, 300))
    for s in sig:
        for x in (s * 2.0 ** e, -s * 2.0 ** e):
            r = _recip(x)
            err = abs(Fraction(r) * Fraction(x) - 1) * Fraction(2) ** 53
            assert err <= 3, (x, r)  # 1.5 units of r are at most 3 u |1 / x|
