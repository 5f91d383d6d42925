"""The fixed-point arithmetic of isum.cuh (sums of products of non-negative numbers) and fix60.cuh (E1 in Q60), compiled for
the host, against exact rational arithmetic."""
import ctypes
import random
from fractions import Fraction

import numpy as np
import pytest

from tests.host_build import compile_host

SOURCE = """
#include "fix60.cuh"
using namespace heat;
// sums over n fours, each four aligned (0) or one by one (1)
extern "C" double dot(int n, const double* a, const double* b, int form) {
    ISum s;
    for (int q = 0; q < n; ++q) {
        double x[4], y[4];
        for (int u = 0; u < 4; ++u) x[u] = a[4 * q + u], y[u] = b[4 * q + u];
        if (form == 0) {
            const Align4 p = align4(x), r = align4(y);
            add_aligned4(s, p.h, p.l, p.E, r.h, r.l, r.E);
        } else {
            Mant p[4], r[4];
            for (int u = 0; u < 4; ++u) p[u] = mant(x[u]), r[u] = mant(y[u]);
            add_each4(s, p, r);
        }
    }
    return s.value();
}
extern "C" long long q60(double z) { return to_q60(z); }
extern "C" double dq60(long long v) { return from_q60(v); }
extern "C" long long mq60(long long a, long long b) { return mul_q60(a, b); }
extern "C" int cls(double z) { return e1_class(z); }
extern "C" long long e1(int c, long long z) { return e1_q60(c, z); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = compile_host(str(tmp_path_factory.mktemp("fixed_point")), SOURCE)
    d, q, i, p = ctypes.c_double, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p
    for name, res, args in (("dot", d, [i, p, p, i]), ("q60", q, [d]), ("dq60", d, [q]), ("mq60", q, [q, q]),
                            ("cls", i, [d]), ("e1", q, [i, q])):
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


def _dot(host, a, b, form):
    a, b = np.ascontiguousarray(a, np.float64), np.ascontiguousarray(b, np.float64)
    assert len(a) % 4 == 0
    return host.dot(len(a) // 4, a.ctypes.data, b.ctypes.data, form)


def _exact(a, b):
    return sum((Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)), Fraction(0))


ULP = Fraction(1, 2**53)


def _dropped(a, b):
    """What the aligned form may drop, per four: three operands' bits below the largest's last place (2^-56 of it each) and
    five units of the product, of which the largest operands' product has at least 2^58."""
    return sum(Fraction(float(a[k:k + 4].max())) * Fraction(float(b[k:k + 4].max())) * Fraction(17, 2**58)
               for k in range(0, len(a), 4))


@pytest.mark.parametrize("span", [0, 3, 40, 400])
@pytest.mark.parametrize("n", [4, 16, 400])
def test_sums_of_products(host, n, span):
    rng = np.random.default_rng(n + span)
    a = rng.uniform(1, 2, n) * 2.0 ** rng.integers(-span, span + 1, n)
    a[rng.random(n) < 0.2] = 0.0
    near = rng.uniform(1, 2, n) * np.repeat(2.0 ** rng.integers(-span, span + 1, n // 4), 4) * 2.0 ** rng.integers(0, 4, n)
    far = rng.uniform(1, 2, n) * 2.0 ** rng.integers(-span, span + 1, n)
    # each addition drops less than 2^-59 of the sum so far, the value is rounded once
    ref = _exact(a, near)
    assert abs(Fraction(_dot(host, a, near, 0)) - ref) <= ref * (ULP + Fraction(n, 2**59)) + _dropped(a, near)
    ref = _exact(a, far)
    assert abs(Fraction(_dot(host, a, far, 1)) - ref) <= ref * (ULP + Fraction(n, 2**59))


def test_zeros_and_the_carry(host):
    z = np.zeros(8)
    assert _dot(host, z, z, 0) == 0.0 and _dot(host, z, z, 1) == 0.0
    # (2 - 2^-52) 1 + 2^-53: all ones, and a half unit above: rounds to the next power of two
    a = np.array([2.0 - 2.0**-52, 2.0**-53, 0.0, 0.0])
    assert _dot(host, a, np.ones(4), 1) == 2.0 and _dot(host, a, np.ones(4), 0) == 2.0


def test_negative_zero(host):
    a = np.array([1.5, -0.0, 3.0, 0.0, -0.0, -0.0, -0.0, -0.0])
    for form in (0, 1):
        assert _dot(host, a, np.array([1.0, 2.0, -0.0, 1.0] * 2), form) == 1.5
        assert _dot(host, np.abs(a), np.array([1.0, -0.0, -0.0, 1.0] * 2), form) == 1.5


# Subnormal operands count at their value, results below the normal range are rounded to its last place (2^-1074).  The
# aligned form's bound is against the largest of a four, at least 2^-1022 here.
@pytest.mark.parametrize("seed", range(20))
def test_subnormals(host, seed):
    rng = np.random.default_rng(seed)
    tiny = Fraction(1, 2**1074)
    n = 16
    sub = rng.integers(1, 2**52, n).astype(np.float64) * 2.0**-1074 * 2.0 ** -rng.integers(0, 50, n)
    sub[sub == 0.0] = 2.0**-1074
    w = rng.uniform(0.5, 1.0, n)
    for a, b in ((sub, w), (w, sub)):
        ref = _exact(a, b)
        assert abs(Fraction(_dot(host, a, b, 1)) - ref) <= ref * (ULP + Fraction(n, 2**59)) + tiny / 2
        lost = n // 4 * Fraction(17, 2**58) * Fraction(1, 2**1022)
        assert abs(Fraction(_dot(host, a, b, 0)) - ref) <= ref * (ULP + Fraction(n, 2**59)) + lost + tiny / 2
    # normal operands, a subnormal product
    a, b = w * 2.0**-600, rng.uniform(0.5, 1.0, n) * 2.0 ** -rng.integers(421, 480, n)
    ref = _exact(a, b)
    assert abs(Fraction(_dot(host, a, b, 1)) - ref) <= ref * (ULP + Fraction(n, 2**59)) + tiny / 2
    assert _dot(host, np.full(4, 2.0**-600), np.full(4, 2.0**-474), 1) == 2.0**-1072
    assert _dot(host, np.full(4, 2.0**-600), np.full(4, 2.0**-600), 1) == 0.0


def test_overflow(host):
    big = np.full(8, 2.0**512)
    for form in (0, 1):
        assert _dot(host, big, big, form) == np.inf
        assert _dot(host, big[:4], big[:4] * np.array([0.125, 0.125, 0.125, 0.0625]), form) == 7 * 2.0**1020
        assert _dot(host, big[:4], big[:4] * 0.25, form) == np.inf  # four quarters of 2^1024


def _e1_exact(z, bits=200):
    """E1(z) = sum z^k / (k+1)! for z in Q60, as an integer times 2^-bits."""
    s, t, k = 0, 1 << bits, 0
    while t:
        s += t
        k += 1
        t = (abs(t) * abs(z) >> 60) // (k + 1) * (1 if z >= 0 or k % 2 == 0 else -1)
    return s


# The trailing stage loses at most three of its units a step (coefficient, product, z's low bits), the leading one three of
# Q60: for |z| <= 1, the worst, 7 x 3 x 4 + 10 x 3 = 114 of Q60, 2^-53.2, against E1 >= 1 for z >= 0; for z < 0 the steps'
# losses alternate, half of it against E1 >= 0.63.
@pytest.mark.parametrize("c,edge", [(3, 1 / 16), (2, 1 / 4), (1, 1.0)])
def test_e1_series(host, c, edge):
    rng = random.Random(c)
    below = np.nextafter(edge, 0.0)
    zs = [0.0, 2.0**-70, -(2.0**-70), 1e-9, below, -below] + [rng.uniform(-edge, edge) for _ in range(300)]
    for z in zs:
        assert host.cls(z) >= c
        q = host.q60(z)
        assert q == int(Fraction(z) * 2**60)  # towards zero
        assert abs((host.e1(c, q) << 140) - _e1_exact(q)) <= _e1_exact(q) >> 53
    assert host.cls(edge) == c - 1 and host.cls(-edge) == c - 1


def test_q60_products_and_rounding(host):
    rng = random.Random(7)
    for _ in range(2000):
        a, b = rng.randrange(-2**61 + 1, 2**61), rng.randrange(-2**61 + 1, 2**61)
        if rng.random() < 0.3:
            b >>= rng.randrange(60)
        if abs(a * b) >> 120 < 2:
            assert abs((host.mq60(a, b) << 60) - a * b) <= 2 << 60
        v = abs(a) >> rng.randrange(61) or 1
        assert abs(Fraction(host.dq60(v)) * 2**60 - v) <= v * ULP
