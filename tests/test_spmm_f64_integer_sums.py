"""CPU pin of the FP64 SpMM's aligned integer sums, independent of the GPU code: the kernel adds, of
every four values of a row's run, one in FP64 and three as 64-bit integers.  The integer part is
restated here in exact integers and checked against exact sums.

Restated: a sum holds the integer a in units of 2^(e - 57), e the largest exponent so far.  Before a
group of three values is added e rises to the largest of theirs and a is shifted right (floor).  A
value's significand with the leading one (53 bits, shifted up by 5) is shifted right by its distance to e
and, where it is negative, its bits are inverted (-t - 1) and the group's count of negative values is
added back.  After eight groups a goes to FP64 in one rounding.

Stated error between two conversions: below 2^-52 of the largest value (24 values and 8 shifts of at
most one unit of 2^-57 each), and none where no bit is dropped: whole numbers come out exact."""
from fractions import Fraction

import numpy as np
import pytest

MASK = (1 << 64) - 1


def _signed(x):
    x &= MASK
    return x - (1 << 64) if x >> 63 else x


def fx_align(x, e):
    u = int(np.float64(x).view(np.uint64))
    ev = (u >> 52) & 0x7FF
    t = (((u & ((1 << 52) - 1)) | ((1 << 52) if ev else 0)) << 5) >> (e - ev)
    return _signed(t ^ (MASK if u >> 63 else 0))


def fx_add3(a, e, xs, count_signs=True):
    us = [int(np.float64(x).view(np.uint64)) for x in xs]
    top = max([e] + [(u >> 52) & 0x7FF for u in us])
    a >>= top - e
    a += sum(fx_align(x, top) for x in xs)
    if count_signs:
        a += sum(u >> 63 for u in us)
    assert -(1 << 63) <= a < 1 << 63
    return a, top


def group_sum(values, count_signs=True):
    """The exact value that up to eight groups of three leave before the conversion to FP64."""
    a, e = 0, 0
    assert len(values) % 3 == 0 and len(values) <= 24
    for i in range(0, len(values), 3):
        a, e = fx_add3(a, e, values[i:i + 3], count_signs)
    return Fraction(a) * Fraction(2) ** (e - 1080)


def _exact(values):
    return sum((Fraction(float(v)) for v in values), Fraction(0))


def _rows(seed):
    r = np.random.default_rng(seed)
    v = r.standard_normal(24)
    yield "normal", v
    yield "one sign", -np.abs(v) - 1.0
    yield "wide", np.ldexp(v, r.integers(-900, 900, 24))
    yield "rising", np.ldexp(v, 2 * np.arange(24))
    yield "rising by more than 57", np.ldexp(v, 60 * (np.arange(24) // 3))
    yield "falling", np.ldexp(v, -3 * np.arange(24))
    yield "largest", np.full(24, -np.nextafter(2.0, 1.0))
    yield "cancel", np.concatenate([v[:12], -v[:12]])


@pytest.mark.parametrize("seed", range(20))
def test_error_between_conversions(seed):
    for name, v in _rows(seed):
        err = abs(group_sum(v) - _exact(v))
        assert err < Fraction(2) ** -52 * Fraction(float(np.abs(v).max())), name


@pytest.mark.parametrize("seed", range(20))
def test_whole_numbers_are_exact(seed):
    r = np.random.default_rng(seed)
    for v in (np.where(r.random(24) < 0.5, -1.0, 1.0), r.integers(-1000, 1001, 24).astype(float),
              r.integers(-2 ** 52, 2 ** 52, 24).astype(float), np.where(r.random(24) < 0.5, -0.0, -3.0),
              np.tile([1.0, -1.0, 0.0], 8)):
        assert group_sum(v) == _exact(v)


def test_the_pin_sees_a_lost_unit():
    """Without the count of negative values every one of them is a unit low: +1 -1 no longer cancels."""
    v = np.tile([1.0, -1.0, -1.0, 1.0, 1.0, -1.0], 4)
    assert group_sum(v) == 0
    assert group_sum(v, count_signs=False) == -12 * Fraction(2) ** -57
