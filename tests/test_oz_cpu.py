"""The digit splitting behind the tensor-core Schur products (kkt_oz.cuh), its
host forms against exact rational arithmetic: digits and their value, the
digit sums' bounds, and the dot product of two rows against the exact one and
against a chain of FP64 FMAs."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
FP64_ROW = 1 << 20


@pytest.fixture(scope="module")
def lib():
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "liboz_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so,
                           os.path.join(HERE, "csrc", "oz_host.cpp")])
    L = ctypes.CDLL(so)
    L.oz_value.restype = L.oz_to_double.restype = L.oz_dot.restype = ctypes.c_double
    L.oz_value.argtypes = [ctypes.c_ulonglong, ctypes.c_int]
    L.oz_to_double.argtypes = [ctypes.c_longlong, ctypes.c_int]
    vp = ctypes.c_void_p
    L.oz_row.argtypes = [vp, ctypes.c_int, vp]
    L.oz_dot.argtypes = [vp, ctypes.c_int, vp, ctypes.c_int, ctypes.c_int, vp]
    return L


def row(lib, z):
    z = np.ascontiguousarray(z, dtype=np.float64)
    u = np.zeros(len(z), dtype=np.uint64)
    return lib.oz_row(z.ctypes.data, len(z), u.ctypes.data), u


def dot(lib, a, b):
    (fa, ua), (fb, ub) = row(lib, a), row(lib, b)
    p = np.zeros(7, dtype=np.int64)
    return lib.oz_dot(ua.ctypes.data, fa, ub.ctypes.data, fb, len(a), p.ctypes.data), p, fa, fb


def exact(a, b):
    return sum((Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)), Fraction(0))


def test_digits_and_value(lib):
    rng = np.random.default_rng(1)
    for scale in (0, 1, 8, 40, 300):
        z = rng.normal(size=64) * 2.0 ** rng.integers(-scale, scale + 1, size=64)
        f, u = row(lib, z)
        assert np.abs(z).max() < 2.0 ** f <= 2 * np.abs(z).max()
        for x, v in zip(z, u):
            assert int(v) < 1 << 63
            assert abs(Fraction(lib.oz_value(int(v), f)) - Fraction(float(x))) <= Fraction(2) ** (f - 62)
            if abs(x) >= 2.0 ** (f - 9):  # within 2^-8 of the row's scale: exact
                assert lib.oz_value(int(v), f) == x
    f, u = row(lib, [0.0, -0.0])
    assert f == -1022 and all(lib.oz_value(int(v), f) == 0.0 for v in u)
    f, u = row(lib, [3e-280, -1e-281])  # far below one: split like any other
    assert [lib.oz_value(int(v), f) for v in u] == [3e-280, -1e-281]
    for bad in (np.nan, np.inf, 1e300, 5e-324, 1e-300):
        assert row(lib, [bad, bad / 4])[0] == FP64_ROW


def test_products_below_the_normal_range(lib):
    """Gradual underflow: within the smallest subnormal of the exact product
    (and the split's own bound)."""
    rng = np.random.default_rng(3)
    for s in (-480, -510, -516, -525, -560):
        a, b = rng.normal(size=20) * 2.0 ** s, rng.normal(size=20) * 2.0 ** s
        got, _, fa, fb = dot(lib, a, b)
        x = exact(a, b)
        assert abs(Fraction(got) - x) <= abs(x) / 2**53 + 20 * Fraction(2.0 ** -57.9) * Fraction(2) ** (fa + fb) + \
            Fraction(2) ** -1074


def test_to_double_rounds_to_nearest(lib):
    rng = np.random.default_rng(2)
    for _ in range(3000):
        v = int(rng.integers(-2**62, 2**62)) >> int(rng.integers(0, 62))
        e = int(rng.integers(-800, 800))
        d = Fraction(lib.oz_to_double(v, e))
        x = Fraction(v) * Fraction(2) ** e
        ulp = Fraction(2) ** (max(abs(v).bit_length() - 53, 0) + e)
        assert abs(d - x) <= ulp / 2
    assert lib.oz_to_double(0, 5) == 0.0


@pytest.mark.parametrize("n", [1, 16, 31, 32, 33, 48])
def test_dot_product(lib, n):
    """|error| <= 2^-53 |sum| (one rounding) + n 2^-57.9 2^(fa + fb): the dropped
    digit pairs i + j <= 5 are at most 2^16 (6 2^45 + 5 2^36 + ..) < 2^63.6
    units of 2^-122 per term, the digits' own rounding 2 2^-62. On random rows
    the error is no larger than that of FP64 FMAs (root mean square)."""
    rng = np.random.default_rng(n)
    se = sf = 0.0
    for t in range(60):
        s = 2.0 ** rng.integers(-6, 7, size=n) if t % 3 == 1 else 10.0 ** (-4.0 * np.arange(n) / n) if t % 3 else 1.0
        a, b = rng.normal(size=n) * s, rng.normal(size=n) * s
        got, p, fa, fb = dot(lib, a, b)
        x = exact(a, b)
        unit = Fraction(2) ** (fa + fb)
        assert abs(Fraction(got) - x) <= abs(x) / 2**53 + n * unit * Fraction(2.0 ** -57.9)
        chain = Fraction(0)
        for u, v in zip(a, b):  # correctly rounded FMA chain
            chain = Fraction(float(chain + Fraction(float(u)) * Fraction(float(v))))
        se += float((Fraction(got) - x) / unit) ** 2
        sf += float((chain - x) / unit) ** 2
    assert se <= 1.05 * sf + 1e-40, (se, sf)


@pytest.mark.parametrize("n", [16, 32, 48])
def test_digit_sums_stay_exact_in_fp32(lib, n):
    """Largest digits everywhere: the sums for i + j >= 8 stay below 2^24
    whatever the digits; the two lowest ones exceed it only beyond K = 36 and
    weigh 2^-59 of the rows' scales."""
    z = np.full(n, -(256.0 / 511.0))  # every digit -256 but the leading one
    _, p, _, _ = dot(lib, z, z)
    assert (np.abs(p[2:]) < 2**24).all(), p
    assert (np.abs(p) <= 7 * n * 2**16).all()
