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
