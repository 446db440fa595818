"""Where the integer arithmetic of csrc/at_fixed.cuh could lose what FP64 keeps:
smoothness indicators that are zero, eps of any size, subnormal numbers."""
import math
from fractions import Fraction

import numpy as np
import pytest

from test_fixed_cpu import D1, D2, _call, _weno_exact, lib, soft  # noqa: F401  (fixtures)


def _weno(L, c, q, eps):
    c, q = np.ascontiguousarray(c, dtype=np.float64), np.ascontiguousarray(q, dtype=np.float64)
    return L.weno(c.ctypes.data, q.ctypes.data, 3.0 * eps)


FLAT = [(0, 0, 0, 1, 1), (1, 1, 0, 0, 0), (0, 0, 0, 0, 1), (1, 0, 0, 0, 0), (0, 0, 1, 0, 0), (0, 1, -1, 0, 0),
        (0, 0, 0, 1, -0.75)]


@pytest.mark.parametrize("eps", [1e-6, 1e-30, 1e-100, 1e-140])
@pytest.mark.parametrize("amp", [1e-20, 1e-6, 1.0, 1e7, 1e9, 1e20, 1e24])
@pytest.mark.parametrize("family", [0, 1])
def test_weno_sum_beside_a_uniform_state(soft, amp, eps, family):
    """Exactly uniform gas beside a front: one, two or four of the six
    indicators are zero, and eps alone is their denominators.  The bound is
    that of the general inputs, 32 2^-53 of the largest difference."""
    for shape in FLAT:
        f, zero = amp * np.array(shape, dtype=np.float64), np.zeros(5)
        c, q = (f, zero) if family == 0 else (zero, f)
        got = _weno(soft, c, q, eps)
        assert math.isfinite(got)
        assert abs(Fraction(got) - _weno_exact(c, q, eps)) <= 32 * Fraction(float(np.abs(f).max())) / 2 ** 53


def test_weno_sum_at_the_ends_of_eps(soft):
    """eps = 0 leaves a zero indicator to decide alone, as in FP64; an eps that
    is no number, or infinite, makes the flux no number."""
    zero = np.zeros(5)
    for amp in (1e-200, 1e-170, 1e-20, 1.0, 1e20):
        for shape in ((0, 0, 0, 1, 1), (1, 1, 0, 0, 0), (0, 0, 1, 3, 4)):
            f = amp * np.array(shape, dtype=np.float64)
            if any(d == 0 for d in _indicator_counts(f)):
                continue  # two zero indicators of one reconstruction: 0 / 0
            assert abs(Fraction(_weno(soft, f, zero, 0.0)) - _weno_exact(f, zero, 0.0)) <= 32 * Fraction(4 * amp) / 2 ** 53
    for bad in (math.nan, math.inf):
        assert math.isnan(_weno(soft, np.ones(5), zero, bad))
        assert math.isnan(_weno(soft, np.array([1.0, -2.0, 3.0, 0.5, 1.0]), zero, bad))


def _indicator_counts(f):
    """for both reconstructions the exact denominator with eps = 0 and q = 0"""
    out = []
    for a in (f[[0, 1, 2, 3]], -f[[4, 3, 2, 1]]):
        a = [Fraction(float(v)) for v in a]
        s = [a[1] - a[0], a[2] - a[1], a[3] - a[2]]
        d = [s[0] * (Fraction(4, 3) * s[0] + a[1]) + a[1] ** 2, s[1] * (Fraction(4, 3) * s[1] + a[1]) + a[1] ** 2,
             s[2] * (Fraction(4, 3) * s[2] - a[2]) + a[2] ** 2]
        e = [x * x for x in d]
        out.append(e[1] * (3 * e[0] + e[2]) + 6 * e[0] * e[2])
    return out


@pytest.mark.parametrize("h", (1, 2, 3))
@pytest.mark.parametrize("k", (1, 2))
def test_differences_of_subnormal_numbers(lib, k, h):
    """No worse than a chain of FMAs may be: 2H + 1 roundings of partial sums,
    each half a unit of the sum's last place."""
    taps = (D1 if k == 1 else D2)[h]
    rng = np.random.default_rng(8)
    rows = [np.eye(2 * h + 1)[i] * v for i in range(2 * h + 1) for v in (5e-324, 1e-310, 2e-308, 3e-308)]
    rows += [np.ldexp(rng.integers(-(1 << 53), 1 << 53, 2 * h + 1).astype(np.float64), -1074 - s)
             for s in (0, 1, 2, 10, 30, 50) for _ in range(40)]
    for f in rows:
        exact = sum((t * Fraction(float(v)) for t, v in zip(taps, f)), Fraction(0))
        got = _call(lib, k, f)
        big = Fraction(float(np.abs(f).max()))
        room = sum(abs(t) for t in taps) * big / 2 ** 53 + Fraction(2) ** -1075
        assert abs(Fraction(got) - exact) <= (2 * h + 1) * room


def test_join_undoes_split(tmp_path):
    import ctypes
    import os
    import subprocess
    from test_fixed_cpu import CSRC
    src, so = tmp_path / "j.cpp", str(tmp_path / "j.so")
    src.write_text('#include "at_fixed.cuh"\nextern "C" double j(double x) { return atk::fx_join(atk::fx_split(x)); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so], check=True)
    f = ctypes.CDLL(so).j
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double]
    for x in (0.0, 5e-324, 1e-310, math.nextafter(2.0 ** -1022, 0), 2.0 ** -1022, 1e-300, 1.0, 1.7e308, math.inf):
        assert f(x) == x and f(-x) == -x
    assert math.isnan(f(math.nan))


def _chain(f, taps):
    """the taps over the values by FMAs, each rounded as FP64 does"""
    x = 0.0
    for t, v in zip(taps, f):
        if t:
            x = float(t * Fraction(float(v)) + Fraction(x))
    return x


def _resolved(h, rng):
    o = np.arange(-h, h + 1)
    for g in (1.0, 1.2, 1.5, 2.0):  # a point, up and down
        for s in (1, -1):
            yield "%g^%d" % (g, s), lambda g=g, s=s: g ** (s * o) * (1 + 0.3 * rng.uniform(0, 1, len(o)))
    for w in (0.1, 0.5, 2.0):
        yield "sine %g" % w, lambda w=w: np.sin(w * o + rng.uniform(0, 6.28))
    yield "ripple", lambda: 1 + 0.01 * np.sin(0.2 * o + rng.uniform(0, 6.28))
    yield "bell", lambda: np.exp(-(o + rng.uniform(0, 6.28)) ** 2 / 50)
    yield "random", lambda: rng.uniform(-1, 1, len(o))


@pytest.mark.parametrize("h", (1, 2, 3))
@pytest.mark.parametrize("k", (1, 2))
def test_rows_of_a_few_binades_are_no_less_accurate_than_fmas(lib, k, h):
    """Mean error against the exact sum, relative to the largest value: at most
    that of the chain of FMAs on the same stencils (and two per cent: with H = 1
    both are one rounding, and a value may be cut)."""
    taps = (D1 if k == 1 else D2)[h]
    rng = np.random.default_rng(12)
    for name, row in _resolved(h, rng):
        ours, fmas = Fraction(0), Fraction(0)
        for _ in range(300):
            f = row()
            exact = sum((t * Fraction(float(v)) for t, v in zip(taps, f)), Fraction(0))
            big = Fraction(float(np.abs(f).max()))
            ours += abs(Fraction(_call(lib, k, f)) - exact) / big
            fmas += abs(Fraction(_chain(f, taps)) - exact) / big
        assert ours <= fmas * Fraction(102, 100), (name, float(ours / fmas))


@pytest.mark.parametrize("h", (1, 2, 3))
@pytest.mark.parametrize("k", (1, 2))
def test_steep_rows_keep_the_absolute_bound(lib, k, h):
    """Values growing up to 10^4 times a point: half an ulp of the result, and a
    unit of 2^-55 of the largest value for every tap."""
    taps = (D1 if k == 1 else D2)[h]
    rng, o = np.random.default_rng(14), np.arange(-h, h + 1)
    for g in (2.7, 4.0, 7.4, 16.0, 64.0, 1e4):
        for i in range(200):
            f = g ** ((1 if i % 2 else -1) * o) * (1 + 0.3 * rng.uniform(0, 1, len(o)))
            exact = sum((t * Fraction(float(v)) for t, v in zip(taps, f)), Fraction(0))
            big = Fraction(float(np.abs(f).max()))
            room = Fraction(32 + sum(abs(t) for t in taps)) * big / 2 ** 55
            assert abs(Fraction(_call(lib, k, f)) - exact) <= abs(exact) / 2 ** 53 + room


def test_large_second_differences(lib):
    """Values of one exponent, nothing cut: half an ulp, and 2^-50 of the largest
    value where the sum does not fit 64 bits."""
    rng = np.random.default_rng(13)
    for _ in range(3000):
        f = rng.uniform(1.0, 2.0, 7) * rng.choice([-1.0, 1.0], 7)
        exact = sum((t * Fraction(float(v)) for t, v in zip(D2[3], f)), Fraction(0))
        assert abs(Fraction(_call(lib, 2, f)) - exact) <= abs(exact) * Fraction(1001, 1000) / 2 ** 53 + Fraction(2) ** -49


def test_weno_sum_of_differences_next_to_the_subnormal_range(soft):
    """Subnormal differences beside small normal ones, and subnormal ones alone;
    eps in proportion.  The general bound, and the result's own last place (a
    result below the normal range is zero)."""
    rng = np.random.default_rng(15)
    for i in range(400):
        c, q = (np.ldexp(rng.uniform(-1, 1, 5), rng.integers(-1030, (-1021, -1005, -980)[i % 3], 5)) for _ in range(2))
        got = Fraction(_weno(soft, c, q, 1e-6))
        big = Fraction(float(max(np.abs(c).max(), np.abs(q).max())))
        exact = _weno_exact(c, q, 1e-6)
        if abs(exact) < Fraction(2) ** -1022:
            assert got == 0 or abs(got - exact) <= 32 * big / 2 ** 53 + Fraction(2) ** -1074
        else:
            assert abs(got - exact) <= 32 * big / 2 ** 53 + Fraction(2) ** -1074
