"""Integer forms of FP64 arithmetic (csrc/ix64.cuh): the kernels' own source
built for the host, against exact rationals and IEEE conversions, at random
operands and at significands next to 1 and 2, unlike sizes, ties, signed zeros
and the ends of the ranges."""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1809_10895_gb300", "csrc")
D, F = C.c_double, C.c_float


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    so = str(tmp_path_factory.mktemp("ix64") / "libix64.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "c", "ix64_host.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    for name, res, args in (("rcp", D, [D, C.c_int]), ("div", D, [D, D, C.c_int]),
                            ("sqrt", D, [D]), ("rcp32", F, [D, C.c_int]), ("add_mul", D, [D, D, D]), ("add", D, [D, D]), ("d2f", F, [D]),
                            ("f2d", D, [F])):
        f = getattr(L, "ix_h_" + name)
        f.restype, f.argtypes = res, args
    return L


def significands(rng, n):
    """Random ones, and those next to 1, to 2 and to a float's neighbours."""
    k = np.arange(1, 9) * 2.0 ** -52
    f = np.arange(1, 5) * 2.0 ** -23
    near = np.concatenate([[1.0], 1.0 + k, 2.0 - k, 1.0 + f, 1.0 + f - 2.0 ** -52, 2.0 - f, 2.0 - f - 2.0 ** -52])
    return np.concatenate([rng.uniform(1.0, 2.0, n), near])


def ulps_off(got, exact):
    """|got - exact| in units of the last place of exact > 0."""
    e = np.frexp(float(exact))[1] - 1
    if Fraction(2) ** int(e) > exact:        # float(exact) rounded up to a power of two
        e -= 1
    return abs(Fraction(got) - exact) / Fraction(2) ** int(e - 52)


# One rounding plus what the 64-bit significand loses: a few units of 2^-63,
# and of a reciprocal e^3 <= 2^-60: below a hundredth of a unit of the last place.
TOL = Fraction(51, 100)


# the estimate may be off by 2^-23 on [1, 2): two units of its last place
@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
def test_reciprocal(lib, ulps):
    rng = np.random.default_rng(3)
    for m in significands(rng, 3000):
        a = float(np.ldexp(m, int(rng.integers(-600, 600))))
        assert ulps_off(lib.ix_h_rcp(a, ulps), 1 / Fraction(a)) <= TOL, (m, ulps)


@pytest.mark.parametrize("ulps", [-2, 0, 2])
def test_quotient(lib, ulps):
    rng = np.random.default_rng(4)
    sig = significands(rng, 3000)
    for m in sig:
        a = float(np.ldexp(m, int(rng.integers(-320, 320))))
        b = float(np.ldexp(rng.choice(sig), int(rng.integers(-320, 320))))
        assert ulps_off(lib.ix_h_div(a, b, ulps), Fraction(a) / Fraction(b)) <= TOL, (a, b)
    for a, b in ((-1.0, 1.0), (1.0, -1.0), (0.0, 1.0), (1.0, 0.0), (np.inf, 1.0), (1.0, np.nan), (2.0 ** -400, 1.0)):
        assert np.isnan(lib.ix_h_div(a, b, ulps))


# s is within 2^-24 of the root, so the step leaves 2^-48 / 2, the float
# arithmetic of the correction 2^-24 (2^-24 + 2^-23): below 2^-45 together.
def test_square_root(lib):
    rng = np.random.default_rng(8)
    for m in significands(rng, 3000):
        a = float(np.ldexp(m, int(rng.integers(-99, 99))))
        assert abs(Fraction(lib.ix_h_sqrt(a)) ** 2 / Fraction(a) - 1) <= 2 * Fraction(1, 2 ** 44), a


# An FP64 reciprocal (0.51 units of its last place) rounded once to FP32.
@pytest.mark.parametrize("ulps", [-2, 0, 2])
def test_fp32_reciprocal(lib, ulps):
    rng = np.random.default_rng(9)
    for m in significands(rng, 3000):
        a = float(np.ldexp(m, int(rng.integers(-100, 100))))
        assert ulps_off(lib.ix_h_rcp32(a, ulps), 1 / Fraction(a)) <= Fraction(2 ** 29) * (Fraction(1, 2) + Fraction(1, 2 ** 20)), a


@pytest.mark.parametrize("spread", [0, 1, 3, 52, 61, 62, 63, 64, 200])
def test_sum_and_scaled_sum(lib, spread):
    rng = np.random.default_rng(spread)
    for m in significands(rng, 300):
        a, b = float(m), float(np.ldexp(rng.choice(significands(rng, 4)), -spread))
        c = float(np.ldexp(rng.choice(significands(rng, 4)), int(rng.integers(-200, 200))))
        for x, y in ((a, b), (b, a)):
            s = Fraction(x) + Fraction(y)
            assert ulps_off(lib.ix_h_add(x, y), s) <= TOL
            assert ulps_off(lib.ix_h_add_mul(x, y, c), s * Fraction(c)) <= TOL


def test_double_to_float(lib):
    rng = np.random.default_rng(5)
    tiny, big = float(np.finfo(np.float32).tiny), float(np.finfo(np.float32).max)
    half = 2.0 ** -24
    v = [float(x) for x in np.ldexp(rng.uniform(1, 2, 2000), rng.integers(-126, 128, 2000))]
    v += [1.0, 1.0 + half, 1.0 + 3 * half, 1.0 + half - 2.0 ** -52, 1.0 + half + 2.0 ** -52, 2.0 - half, tiny, big,
          big * (1 + 2.0 ** -25), big * (1 + 2.0 ** -24), np.ldexp(2.0 - 2.0 ** -52, 127)]
    with np.errstate(over="ignore"):
        for x in v:
            for a in (x, -x):
                assert lib.ix_h_d2f(a) == float(np.float32(a)), a
    for a in (0.0, -0.0, tiny / 2, float(np.nextafter(tiny, 0)), 2.0 ** 128, np.inf, np.nan, 5e-324):
        assert np.isnan(lib.ix_h_d2f(a)) and np.isnan(lib.ix_h_d2f(-a))


def test_float_to_double(lib):
    rng = np.random.default_rng(6)
    fi = np.finfo(np.float32)
    v = np.ldexp(rng.uniform(1, 2, 2000), rng.integers(-126, 128, 2000)).astype(np.float32)
    for x in np.concatenate([v[np.isfinite(v)], np.array([0.0, fi.tiny, fi.max, 1.0], np.float32)]):
        for a in (float(x), -float(x)):
            got = lib.ix_h_f2d(a)
            assert got == a and np.signbit(got) == np.signbit(a)
    for a in (float(fi.tiny) / 2, np.inf, np.nan):
        assert np.isnan(lib.ix_h_f2d(a))
