"""Sums over lanes, warps and CTAs of the float32 sweeps keep the accuracy of float64 sums.

A lane's products are exact as float pairs; adding the lanes must not lose more than a float64 sum does.
With one product per lane the total is rounded once: half an ulp of a float64 for the last rounding, twice that
for the low terms' own, and additions that lose 2^-72 of the partial sums each (fewer than 2^8 in a row).
"""
import ctypes
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_2110_04015_gb300 import binding

pytestmark = pytest.mark.gpu


def _cancelling(n, seed):
    """float32 a, b whose products nearly cancel: sum |a b| is about 1e6 |a^T b|."""
    rs = np.random.RandomState(seed)
    a = rs.standard_normal(n).astype(np.float32)
    b = rs.standard_normal(n).astype(np.float32)
    h = n // 2
    b[h:2 * h] = b[:h]
    a[h:2 * h] = (-a[:h].astype(np.float64) * (1 + 1e-6 * rs.standard_normal(h))).astype(np.float32)
    return a, b


def _exact(a, b):
    s = sum((Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)), Fraction(0))
    t = math.fsum(np.abs(a.astype(np.float64) * b.astype(np.float64)))
    return s, t


def _ptr(v):
    return ctypes.c_void_p(v.ctypes.data)


def _within(got, a, b):
    s, t = _exact(a, b)
    return abs(Fraction(got) - s) <= Fraction(2) ** -52 * abs(s) + Fraction(2) ** -64 * Fraction(t)


@pytest.mark.parametrize("n, chunk", [(9, 9), (32, 32), (126, 18), (1000, 27), (9000, 27), (4001, 32)])
def test_phi_sums_are_as_accurate_as_float64(n, chunk):
    for seed in range(4):
        a, b = _cancelling(n, seed)
        out = (ctypes.c_double * 3)()
        assert binding.lib().ba_test_float_sums(_ptr(a), _ptr(b), n, chunk, out) == 0
        assert _within(out[0], a, b), (seed, out[0])


# |r|^2, r^T z and q^T z: a product per thread, so any n
@pytest.mark.parametrize("n", [1, 126, 128, 129, 9000, 17424, 40000])
def test_update_sums_are_as_accurate_as_float64(n):
    for seed in range(3):
        a, b = _cancelling(n, seed)
        out = (ctypes.c_double * 3)()
        assert binding.lib().ba_test_float_sums(_ptr(a), _ptr(b), n, 32, out) == 0
        assert _within(out[1], a, b), (seed, out[1])


# Q^T z in the one-CTA sweep: a thread per column and subset, up to 20 cameras of 9 rows
@pytest.mark.parametrize("cams", [1, 2, 3, 7, 13, 20])
def test_one_cta_sums_are_as_accurate_as_float64(cams):
    for seed in range(4):
        a, b = _cancelling(9 * cams, seed)
        out = (ctypes.c_double * 3)()
        assert binding.lib().ba_test_float_sums(_ptr(a), _ptr(b), 9 * cams, 32, out) == 0
        assert _within(out[2], a, b), (seed, out[2])
