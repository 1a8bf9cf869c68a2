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
#include <algorithm>
#include <vector>
extern "C" {
// one row: 1 and its fixed-point sum, or 0 where the kernels take FMAs; the sum by
// FMAs.  parts: of the row's slots, each but the first checked in its first five
int row(const double* c, const double* u, int S, int dim, int parts, double* fixed, double* fmas) {
  int mc = 0, mu = 0;
  bool zero = true;
  double sum = 0.0;
  *fmas = 0.0;
  for (int n = 0; n < S; ++n) {
    zero &= c[n] == 0.0;
    mc = std::max(mc, (int)(fx_bits(c[n]) >> 52) & 0x7ff);
    mu = std::max(mu, (int)((fx_bits(u[n]) >> 32) & 0x7fffffff) | ((uint32_t)fx_bits(u[n]) != 0));
    sum += std::fabs(c[n]);
    *fmas = std::fma(c[n], u[n], *fmas);
  }
  const int E = fx_row_exponent(mc, zero, sum), Eu = mu == 0 ? kFxZero : mu >> 20;
  if (E == kFxPlain || (mu != 0 && (Eu < kFxMin || Eu > kFxMax))) return 0;
  FxSum s;
  uint32_t size = 0, all = 0;
  for (int n = 0; n < S; ++n) {
    const FxLimbs q = fx_coef(c[n], E), v = fx_value((int)(fx_bits(u[n]) >> 32), (int)fx_bits(u[n]), Eu);
    s.mac(q, v.hi, v.lo);
    int p = 0;
    while ((p + 1) * S / parts <= n) ++p;
    if (n - p * S / parts < (p == 0 ? 10 : 5)) size += fx_size(q, v.hi);
    all += fx_size(q, v.hi);
  }
  *fixed = fx_scale(s.total(), E, Eu);
  if (E == kFxZero || Eu == kFxZero || size >= fx_sure(dim)) return 1;
  return dim == 3 && parts == 1 && size >= fx_sure(dim) / 4 && all >= fx_sure(dim) / 4 * 5;
}
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


def test_a_split_is_its_coefficient_within_half_a_unit(fx):
    g = np.random.default_rng(1)
    hi, _ = _split(fx, 1.0, 1023)
    unit = Fraction(1, hi << 28)  # of the value 1
    for _ in range(2000):
        c = float(g.standard_normal()) * 2.0 ** -int(g.integers(0, 70))
        E = max(1023, int(np.frexp(c)[1]) + 1022)
        h, l = _split(fx, c, E)
        err = abs(Fraction(h * 2 ** 28 + l) * unit * Fraction(2) ** (E - 1023) - Fraction(c))
        assert 2 * err <= unit * Fraction(2) ** (E - 1023), c


def _row(fx, c, u, dim=2, parts=1):
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    c, u = np.ascontiguousarray(c, float), np.ascontiguousarray(u, float)
    out = np.zeros(2)
    sure = fx.row(p(c), p(u), len(c), dim, parts, p(out), ctypes.c_void_p(out.ctypes.data + 8))
    return bool(sure), out[0], out[1]


def _errors(fx, c, u, dim, parts=1):
    """Certified?, and the errors of the fixed-point sum and of FMAs over the terms' magnitudes."""
    sure, fixed, fmas = _row(fx, c, u, dim, parts)
    t = [Fraction(float(a)) * Fraction(float(b)) for a, b in zip(c, u)]
    exact, size = sum(t), sum(map(abs, t))
    if size == 0:
        return sure, 0.0, 0.0
    return sure, float(abs(Fraction(fixed) - exact) / size), float(abs(Fraction(fmas) - exact) / size)


def _states(x, g):
    S, d = x.shape
    k, ph = 2 * np.pi * (0.5 + g.random((3, d))), 2 * np.pi * g.random(3)
    h = np.linalg.norm(x[1] - x[0])
    axis = g.standard_normal(d)
    axis /= np.linalg.norm(axis)
    yield "smooth", np.sin(x @ k.T + ph).sum(1)
    yield "random", g.standard_normal(S)
    yield "graded", g.standard_normal(S) * 2.0 ** -g.integers(0, 41, S)
    yield "one value", np.where(np.arange(S) == g.integers(S), 1.1 + g.random(), 0.0)
    yield "one near value", np.where(np.arange(S) == g.integers(10), 1.1 + g.random(), 0.0)
    yield "one large value", g.standard_normal(S) * np.where(np.arange(S) == g.integers(S), 1e6, 1.0)
    yield "parabola", ((x - x[0]) @ axis) ** 2
    yield "slow decay", np.exp(-(x @ axis / h))
    yield "decay", 10.0 ** -(x @ axis / h)
    yield "sign change", (x - x[:2].mean(0)) @ axis


@pytest.mark.parametrize("dim,n,p,q1,kind", [(3, 6, 3, 3, "tensor"), (2, 16, 3, 3, "tensor"),
                                             (3, 6, 2, 2, "tensor"), (2, 10, 2, 2, "simplex")])
def test_no_less_accurate_than_fmas(fx, dim, n, p, q1, kind):
    """Rows of gradient and extrapolation coefficients.  Where the fixed-point
    sum is taken, its error is within the bound of FMAs, S 2^-53 of the terms'
    magnitudes, and its rms over a class of states at most 1.05 times the
    FMAs': with one value both round one product, and the dropped products
    of the low limbs add 2^-56.6 rms to 2^-54.2, 2 % of an rms."""
    from tests import helpers as H
    pb = H.make_problem(dim, n, p, q1, jitter=0.15, seed=3, kind=kind)
    o, g = pb.orc, np.random.default_rng(5)
    x = o.xc[:, :dim]
    got = {}
    inner = np.flatnonzero(np.asarray(o.faces()[1]) >= 0)
    for f in g.choice(inner, 14, replace=False):
        rows = o.face_coef(f)[:, :o.S].transpose(0, 2, 1).reshape(-1, o.S)
        for name, u in _states(x[o.face_stencil(f)], g):
            got.setdefault(name, []).extend(_errors(fx, c, u, dim) for c in rows)
    for cell in g.choice(o.nc, 25, replace=False):
        for name, u in _states(x[o.cell_stencil(cell)], g):
            got.setdefault(name, []).extend(_errors(fx, c, u, dim, 1 if dim == 2 else 4) for c in o.cell_ext(cell))
    for name, e in got.items():
        e = np.array(e)
        sure = e[:, 0] > 0
        assert (e[sure, 1] <= (o.S + 1) * 2.0 ** -53).all(), name
        rms = np.sqrt((e[sure, 1:] ** 2).mean(0)) if sure.sum() >= 30 else (0.0, 0.0)
        assert rms[0] <= 1.05 * rms[1], (name, rms)
        if name == "smooth":  # these are to take the fast sums
            assert sure.mean() >= 0.99, (name, sure.mean())


@pytest.mark.parametrize("slots", [1, 9, 16, 127])
@pytest.mark.parametrize("scale", [2.0 ** (555 - 1023), 1.0, 2.0 ** (1559 - 1023)])
def test_largest_sums_and_ends_of_the_range(fx, slots, scale):
    top = np.nextafter(2.0, 0.0)
    alternate = top * (-1.0) ** np.arange(slots)
    for c in (np.full(slots, 1.0), np.full(slots, -top), alternate):
        for u in (np.full(slots, 1.0), np.full(slots, top), alternate, -alternate):
            for a, b in ((scale, 1.0), (1.0, scale), (scale, scale)):
                t = [Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a * c, b * u)]
                sure, fixed, _ = _row(fx, a * c, b * u)
                # scale^2 leaves the range of doubles: the sum's scale alone is checked
                if not (a == b == scale != 1.0):
                    assert sure and abs(Fraction(fixed) - sum(t)) <= (slots + 1) * sum(map(abs, t)) / 2 ** 53


def test_zero_rows_and_zero_values(fx):
    g = np.random.default_rng(2)
    v, zero = g.standard_normal(64), np.zeros(64)
    assert _row(fx, zero, v)[:2] == (True, 0.0)
    assert _row(fx, v, zero)[:2] == (True, 0.0)
    c = zero.copy()
    c[0] = 1.0
    u = np.ones(64)
    u[0] = 0.0
    assert _row(fx, c, u)[1] == 0.0  # 64 zero coefficients with values, one coefficient without
