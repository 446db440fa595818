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
        "double d%d_%d(const double* f) { return atk::fx_d%d<%d>(f + %d); }\n" % (k, h, k, h, h)
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
                   "double terms(const double* p, const double* m) "
                   "{ return atk::fx_weno_terms(p, p[3], p[4], m, m[3], m[4]); }\n"
                   "int one(int f, double x, double* y) { bool ok = true; "
                   "*y = f == 0 ? atk::fx_rcp(x, &ok) : f == 1 ? atk::fx_sqrt(x, &ok) : atk::fx_half(x); return ok; }\n"
                   "double most(double a, double b) { return atk::fx_fmax(a, b); }\n}\n")
    so = str(d / "s.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    L.recip.restype, L.recip.argtypes = ctypes.c_uint64, [ctypes.c_uint64]
    L.terms.restype, L.terms.argtypes = ctypes.c_double, [ctypes.c_void_p, ctypes.c_void_p]
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


def _terms_exact(side):
    d0, d1, d2, x, y = (Fraction(float(v)) for v in side)
    e0, e1, e2 = d0 * d0, d1 * d1, d2 * d2
    den = e1 * (3 * e0 + e2) + 6 * e0 * e2
    return e1 * (2 * e2 * x + 3 * e0 * y) / den, e1 * (2 * e2 * abs(x) + 3 * e0 * abs(y)) / den


def test_weno_terms_against_the_exact_quotients(soft):
    """Seven products of 57 or more bits, three sums and a reciprocal: below
    2 ulps of the terms' size; the FP64 sequence had 16 roundings of half an
    ulp each."""
    rng = np.random.default_rng(9)
    for i in range(4000):
        amp = 10.0 ** rng.uniform(-9, 4)
        sides = []
        for _ in range(2):
            s0, s1, s2, a2 = amp * rng.uniform(-1, 1, 4) * 10.0 ** rng.uniform(-4 if i % 2 else 0, 0, 4)
            a3 = a2 + s1
            d = [s * (4 / 3 * s + a) + a * a + 1e-6 for s, a in ((s0, a2), (s1, a2), (s2, -a3))]
            sides.append(np.array(d + [s0 - s1, s1 - s2]))
        got = Fraction(soft.terms(sides[0].ctypes.data, sides[1].ctypes.data))
        (tp, sp), (tm, sm) = map(_terms_exact, sides)
        assert abs(got - tp - tm) <= 2 * (sp + sm) / 2 ** 53
    flat = np.array([1e-12, 1e-12, 1e-12, 0.0, -0.0])
    assert soft.terms(flat.ctypes.data, flat.ctypes.data) == 0.0
    for bad in (np.zeros(5), np.array([1.0, math.nan, 1.0, 0.0, 0.0]), np.array([1.0, math.inf, 1.0, 0.0, 0.0])):
        assert math.isnan(soft.terms(bad.ctypes.data, bad.ctypes.data))
        if bad[1] != 0.0:
            assert math.isnan(soft.terms(flat.ctypes.data, bad.ctypes.data))
