"""The fixed-point arithmetic of the default precision as the library has it
(csrc/fixed_point.cuh, compiled for the host), against exact rationals."""
from __future__ import annotations

import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2601_18417_gb300 import build as B

SHIM = r"""
#include "fixed_point.cuh"
using namespace hofv;
extern "C" {
void split(double c, int E, long long* out) { FxLimbs q = fx_coef(c, E); out[0] = q.hi; out[1] = q.lo; }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "shim.cpp").write_text(SHIM)
    so = os.path.join(str(d), "shim.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{B.CSRC}",
                    "-x", "c++", str(d / "shim.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _split(fx, c, E):
    out = (ctypes.c_longlong * 2)()
    fx.split(ctypes.c_double(c), E, out)
    return out[0], out[1]


@pytest.mark.parametrize("E", [555, 1023, 1560])
def test_zero_and_far_smaller_coefficients_have_no_limbs(fx, E):
    big = 2.0 ** (E - 1023)
    for c in (0.0, -0.0, big * 2.0 ** -70, -big * 2.0 ** -65, 5e-324, -1e-310):
        assert _split(fx, c, E) == (0, 0), c
    hi, lo = _split(fx, big, E)
    assert hi > 0 and lo == 0 and _split(fx, -big, E) == (-hi, 0)


def test_a_split_is_its_coefficient_within_one_unit(fx):
    g = np.random.default_rng(1)
    hi, _ = _split(fx, 1.0, 1023)
    unit = Fraction(1, hi << 28)  # of the value 1
    for _ in range(2000):
        c = float(g.standard_normal()) * 2.0 ** -int(g.integers(0, 70))
        E = max(1023, int(np.frexp(c)[1]) + 1022)
        h, l = _split(fx, c, E)
        err = abs(Fraction(h * 2 ** 28 + l) * unit * Fraction(2) ** (E - 1023) - Fraction(c))
        assert err < unit * Fraction(2) ** (E - 1023), c
