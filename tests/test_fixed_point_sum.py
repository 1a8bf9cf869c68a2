"""Host-side pin of the fixed-point sums of the default precision: the split of
coefficients and values into 28-bit limbs as the kernels do it (csrc/residual.cu,
fx_coef and fx_value), in exact integers, against rational arithmetic."""
from fractions import Fraction
import struct

import numpy as np
import pytest

FX_MIN, FX_MAX, MAX_S = 540, 1560, 127


def _bits(x):
    b = struct.unpack("<Q", struct.pack("<d", x))[0]
    return b >> 63, (b >> 52) & 0x7ff, (b & ((1 << 52) - 1)) | (1 << 52)


def _coef(c, E):
    s, e, m = _bits(c)
    sh = min(E - e, 55)
    top = (m << 11) & ((1 << 64) - 1)               # the significand at the top of 64 bits
    hi = (top >> 32) >> (sh + 4) if sh + 4 < 32 else 0
    lo = (top >> (sh + 8)) & 0xfffffff
    return (-hi, -lo) if s else (hi, lo)


def _value(u, E):
    s, e, m = _bits(u)
    v = (((m << 3) >> min(E - e, 63)) + 1) >> 1
    v = -v if s else v
    hi = (v + (1 << 27)) >> 28
    return hi, v - (hi << 28)


def _exp(a):
    return max(FX_MIN, max(_bits(x)[1] for x in a))


def _sum(c, u):
    Ec, Eu = _exp(c), _exp(u)
    hh = x = 0
    for a, b in zip(c, u):
        ch, cl = _coef(a, Ec)
        uh, ul = _value(b, Eu)
        assert abs(ch) < 1 << 28 and abs(cl) < 1 << 28
        assert abs(uh) <= 1 << 27 and -(1 << 27) <= ul < 1 << 27
        hh += ch * uh
        x += ch * ul + cl * uh
        assert abs(hh) < 1 << 63 and abs(x) + (1 << 27) < 1 << 63
    t = hh + ((x + (1 << 27)) >> 28)
    assert abs(t) < 1 << 63
    return Fraction(t) * Fraction(2) ** (Ec + Eu - 2099)


def _check(c, u):
    exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(c, u))
    # a slot: a coefficient below its place by 2^-55 of the largest (truncated), a
    # value by 2^-54.. of a unit, the low limbs' product; the sum's own 2^-55
    bound = Fraction(len(c) + 1) * Fraction(max(abs(np.asarray(c)))) * Fraction(max(abs(np.asarray(u)))) / 2 ** 53
    assert abs(_sum(c, u) - exact) <= bound


@pytest.mark.parametrize("slots", [1, 2, 16, 65, MAX_S])
def test_random_rows(slots):
    g = np.random.default_rng(slots)
    for spread in (0, 8, 70):
        c = g.standard_normal(slots) * 2.0 ** -g.integers(0, spread + 1, slots)
        u = g.standard_normal(slots) * 2.0 ** -g.integers(0, spread + 1, slots)
        _check(list(c), list(u))
        c[:: 2] = 0.0
        _check(list(c), list(u))


@pytest.mark.parametrize("c,u", [(np.nextafter(2.0, 0.0), np.nextafter(2.0, 0.0)), (1.0, 1.0),
                                 (-np.nextafter(2.0, 0.0), np.nextafter(2.0, 0.0)), (1.0, -1.0)])
def test_largest_sums_do_not_overflow(c, u):
    _check([float(c)] * MAX_S, [float(u)] * MAX_S)


def test_ends_of_the_range():
    lo, hi = 2.0 ** (FX_MIN - 1023), 2.0 ** (FX_MAX - 1023)
    for a in (lo, hi):
        for b in (lo, hi):
            _check([a, -1.5 * a, a / 3], [b, b / 7, -1.25 * b])
    # the scales of the sums stay normal numbers
    assert 0 < 1023 + 2 * FX_MIN - 2099 and 1023 + 2 * FX_MAX - 2099 < 2047
