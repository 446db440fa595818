"""The integer arithmetic of csrc/at_fixed.cuh, compiled for the host: it is
the device code's own source, so what holds here holds in the kernels."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_01133_gb300", "csrc")
D1 = {1: [-1, 0, 1], 2: [1, -8, 0, 8, -1], 3: [-1, 9, -45, 0, 45, -9, 1]}
D2 = {1: [1, -2, 1], 2: [-1, 16, -30, 16, -1], 3: [2, -27, 270, -490, 270, -27, 2]}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src = d / "f.cpp"
    src.write_text('#include "at_fixed.cuh"\nextern "C" {\n' + "".join(
        "double d%d_%d(const double* f) { return atk::fx_d%d<%d>(atk::FxDoubles{f + %d}); }\n" % (k, h, k, h, h)
        for k in (1, 2) for h in (1, 2, 3)) + "}\n")
    so = str(d / "f.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    for k in (1, 2):
        for h in (1, 2, 3):
            f = getattr(L, "d%d_%d" % (k, h))
            f.restype, f.argtypes = ctypes.c_double, [ctypes.c_void_p]
    return L


def _call(lib, k, f):
    f = np.ascontiguousarray(f, dtype=np.float64)
    return getattr(lib, "d%d_%d" % (k, (len(f) - 1) // 2))(f.ctypes.data)


def _rows(h, rng):
    n = 2 * h + 1
    x = np.arange(n)
    for e in (-900, -30, 0, 30, 900):
        s = math.ldexp(1.0, e)
        yield s * (1.0 + 0.01 * np.sin(0.2 * x + rng.uniform(0, 6)))   # about the binade's edge
        yield s * np.sin(0.15 * x + rng.uniform(0, 6))                 # through zero
        yield s * rng.uniform(1.5, 1.9, n)                             # one exponent
        yield s * rng.uniform(-1, 1, n)                                # no smoothness
        yield s * np.ldexp(rng.uniform(-1, 1, n), rng.integers(-70, 70, n))  # no common scale
        yield s * np.where(x % 2, 1.0, -1.0) * (2.0 - 2.0 ** -52)      # the largest differences there are


@pytest.mark.parametrize("h", (1, 2, 3))
@pytest.mark.parametrize("k", (1, 2))
def test_differences_against_the_exact_sum(lib, k, h):
    """Never worse than a chain of FMAs may be (2H + 1 roundings of partial
    sums); and where second differences are moderate half an ulp of the
    result plus the cut of every value."""
    taps = (D1 if k == 1 else D2)[h]
    weight = sum(abs(t) for t in taps)
    rng = np.random.default_rng(3)
    for _ in range(200):
        for f in _rows(h, rng):
            exact = sum((t * Fraction(float(v)) for t, v in zip(taps, f)), Fraction(0))
            big = Fraction(float(np.abs(f).max()))
            got = Fraction(_call(lib, k, f))
            err = abs(got - exact)
            assert err <= (2 * h + 1) * weight * big / 2 ** 53
            smooth = k == 1 or h < 3 or float(np.abs(np.diff(f, 2)).max()) < 0.05 * float(big)
            if smooth:
                assert err <= abs(got) / 2 ** 53 + weight * big / 2 ** 55


@pytest.mark.parametrize("h", (1, 2, 3))
@pytest.mark.parametrize("k", (1, 2))
def test_zeros_specials_and_the_ends_of_the_range(lib, k, h):
    n = 2 * h + 1
    assert _call(lib, k, np.where(np.arange(n) % 2, 0.0, -0.0)) == 0.0
    assert _call(lib, k, np.full(n, 0.3)) == 0.0
    for bad in (math.inf, -math.inf, math.nan):
        f = np.ones(n)
        f[h + 1] = bad
        assert not math.isfinite(_call(lib, k, f))
    tiny = np.zeros(n)
    tiny[h + 1] = 5e-324
    assert 0.0 <= abs(_call(lib, k, tiny)) < 1e-300
    huge = np.full(n, 1e300)
    huge[0] = 1.5e300
    taps = (D1 if k == 1 else D2)[h]
    assert _call(lib, k, huge) == pytest.approx(taps[0] * 0.5e300, rel=1e-12)
    # overflow is an infinity, as in FP64
    top = np.where(np.arange(n) < h, -1.7e308, 1.7e308)
    assert math.isinf(_call(lib, 1, top))


@pytest.fixture(scope="module")
def soft(tmp_path_factory):
    d = tmp_path_factory.mktemp("soft")
    src = d / "s.cpp"
    src.write_text('#include "at_fixed.cuh"\nextern "C" {\n'
                   "uint64_t recip(uint64_t m) { return atk::fx_recip(m); }\n"
                   "double weno(const double* c, const double* q, double eps3) "
                   "{ return atk::fx_weno_sum(c, q, atk::fx_unpack(eps3)); }\n"
                   "int one(int f, double x, double* y) { bool ok = true; "
                   "*y = f == 0 ? atk::fx_rcp(x, &ok) : f == 1 ? atk::fx_sqrt(x, &ok) : atk::fx_half(x); return ok; }\n"
                   "double most(double a, double b) { return atk::fx_fmax(a, b); }\n}\n")
    so = str(d / "s.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    L.recip.restype, L.recip.argtypes = ctypes.c_uint64, [ctypes.c_uint64]
    L.weno.restype, L.weno.argtypes = ctypes.c_double, [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double]
    L.one.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_void_p]
    L.most.restype, L.most.argtypes = ctypes.c_double, [ctypes.c_double, ctypes.c_double]
    return L


def _one(L, f, x):
    y = ctypes.c_double()
    return bool(L.one(f, x, ctypes.byref(y))), y.value


def test_reciprocal_root_half_and_maximum(soft):
    """Half an ulp and 2^-58 relative, that is 0.52 ulp; everything outside
    the normal range is handed back."""
    rng = np.random.default_rng(6)
    xs = [math.ldexp(float(m), int(e)) for m, e in zip(rng.uniform(1, 2, 4000), rng.integers(-1020, 1020, 4000))]
    for e in (-1, 0, 1, 2):  # both sides of a power of two, of both parities
        xs += [math.ldexp(1.0, e) * (1 + i * 2.0 ** -52) for i in range(-40, 41)]
    for x in xs:
        ok, r = _one(soft, 0, -x)
        assert ok and abs(Fraction(r) + 1 / Fraction(x)) <= Fraction(math.ulp(r)) * 52 / 100
        ok, r = _one(soft, 1, x)
        lo, hi = Fraction(r) - Fraction(math.ulp(r)) * 52 / 100, Fraction(r) + Fraction(math.ulp(r)) * 52 / 100
        assert ok and lo * lo <= Fraction(x) <= hi * hi
        assert _one(soft, 2, x)[1] == 0.5 * x
    for x in (0.0, -0.0, math.inf, -math.inf, math.nan, 1e-310):
        assert not _one(soft, 0, x)[0] and not _one(soft, 1, x)[0]
        h = _one(soft, 2, x)[1]
        assert h == (0.0 if abs(x) < 1 else 0.5 * x) or h != h
    assert not _one(soft, 1, -1.0)[0] and not _one(soft, 0, 1.7e308)[0]
    for a in (0.0, 1.0, 2.0, math.inf, math.nan):
        for b in (0.0, 1.0, 2.0, math.inf, math.nan):
            want = b if a != a else a if b != b else max(a, b)
            got = soft.most(a, b)
            assert got == want or (got != got and want != want)


def test_integer_reciprocal(soft):
    rng = np.random.default_rng(5)
    top = 1 << 63
    ms = [top + i for i in range(600)] + [(1 << 64) - 1 - i for i in range(600)] + [top | 1 << i for i in range(63)]
    ms += [top | int(v) for v in rng.integers(0, top, 20000, dtype=np.uint64)]
    for m in ms:
        r = soft.recip(m)
        assert 1 << 62 <= r <= 1 << 63
        assert abs(r * m - (1 << 126)) <= 1 << 66


def _weno_exact(c, q, eps):
    """six times (the weighted corrections) minus the middle second differences, both signs, exactly"""
    c, q = [Fraction(float(v)) for v in c], [Fraction(float(v)) for v in q]
    total = Fraction(0)
    for a in ([q[j] + c[j] for j in (0, 1, 2, 3)], [q[j] - c[j] for j in (4, 3, 2, 1)]):
        s0, s1, s2 = a[1] - a[0], a[2] - a[1], a[3] - a[2]
        e = Fraction(eps)
        d0 = s0 * (Fraction(4, 3) * s0 + a[1]) + a[1] ** 2 + e
        d1 = s1 * (Fraction(4, 3) * s1 + a[1]) + a[1] ** 2 + e
        d2 = s2 * (Fraction(4, 3) * s2 - a[2]) + a[2] ** 2 + e
        e0, e1, e2 = d0 ** 2, d1 ** 2, d2 ** 2
        den = e1 * (3 * e0 + e2) + 6 * e0 * e2
        total += (2 * e1 * e2 * (s0 - s1) + 3 * e0 * e1 * (s1 - s2)) / den - s1
    return total


def test_weno_sum_against_the_exact_weights(soft):
    """Every difference is cut below 2^-57 of the largest; a cut of one unit
    moves the sum by at most some tens of units (four taps of up to 8 with
    weights up to 2, and the weights' own response, of the same size), two
    signs: 32 2^-53 of the largest difference bounds it with room."""
    rng = np.random.default_rng(9)
    for i in range(4000):
        amp = 10.0 ** rng.uniform(-12, 6)
        kind = i % 4
        c, q = amp * rng.uniform(-1, 1, 5), amp * rng.uniform(-1, 1, 5)
        if kind == 1:    # smooth
            c, q = amp * (1 + 0.1 * np.sin(0.2 * np.arange(5) + rng.uniform(0, 6))), 0.7 * amp * np.cos(0.1 * np.arange(5))
        elif kind == 2:  # a front at one end, quiet at the other
            c, q = c * 10.0 ** -np.arange(0, 15, 3.0), q * 10.0 ** -np.arange(0, 15, 3.0)
        elif kind == 3:  # one family only
            q = np.zeros(5)
        got = Fraction(soft.weno(c.ctypes.data, q.ctypes.data, 3e-6))
        big = Fraction(float(max(np.abs(c).max(), np.abs(q).max())))
        assert abs(got - _weno_exact(c, q, 1e-6)) <= 32 * big / 2 ** 53
    zero = np.zeros(5)
    assert soft.weno(zero.ctypes.data, zero.ctypes.data, 3e-6) == 0.0
    assert math.isnan(soft.weno(zero.ctypes.data, zero.ctypes.data, 0.0))
    for bad in (math.nan, math.inf, -math.inf):
        for j in range(5):
            f = np.ones(5)
            f[j] = bad
            assert math.isnan(soft.weno(f.ctypes.data, zero.ctypes.data, 3e-6))
            assert math.isnan(soft.weno(zero.ctypes.data, f.ctypes.data, 3e-6))
    for amp in (1e-300, 1e250):  # no intermediate leaves its range
        f = amp * np.array([1.0, -2.0, 3.0, 0.5, 1.0])
        big = Fraction(3 * amp)
        assert abs(Fraction(soft.weno(f.ctypes.data, zero.ctypes.data, 3e-6)) - _weno_exact(f, zero, 1e-6)) <= 32 * big / 2 ** 53
