"""Integer sums of doubles (csrc/ix_sum.cuh): the kernels' own source built for
the host, against exact rational sums, over terms of like and of unlike size,
cancelling terms, subnormals, and infinities and NaN."""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1809_10895_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    so = str(tmp_path_factory.mktemp("ixsum") / "libixsum.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "c", "ixsum_host.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    DP = C.POINTER(C.c_double)
    L.ix_sum32.restype, L.ix_sum32.argtypes = C.c_double, [DP, C.c_int]
    L.ix_sum_seven.restype, L.ix_sum_seven.argtypes = C.c_double, [DP]
    return L, DP


@pytest.fixture(scope="module")
def sum32(lib):
    L, DP = lib
    return lambda v: L.ix_sum32(v.ctypes.data_as(DP), v.size)


# A term loses less than 2^-77 of the largest exponent's unit, 32 of them less
# than 2^-72; the result is rounded once.
@pytest.mark.parametrize("spread", [0, 3, 24, 26, 52, 80, 300, 1500])
@pytest.mark.parametrize("n", [1, 2, 31, 32])
def test_against_exact_sums(sum32, n, spread):
    rng = np.random.default_rng(1000 * spread + n)
    for _ in range(200):
        v = np.ldexp(rng.uniform(1, 2, n) * rng.choice([-1.0, 1.0], n), rng.integers(-spread // 2, spread // 2 + 1, n))
        if n > 2 and rng.random() < 0.3:
            v[0] = -v[1:].sum()
        exact = sum(Fraction(float(x)) for x in v)
        got = Fraction(sum32(v))
        top = Fraction(2) ** int(np.frexp(np.abs(v)).__getitem__(1).max() - 1)
        assert abs(got - exact) <= abs(exact) / 2 ** 53 + top / 2 ** 72 * (1 + Fraction(1, 2 ** 52))


def test_edges(sum32):
    tiny, big = 5e-324, np.finfo(float).max
    for v, want in (([0.0, -0.0], 0.0), ([tiny] * 32, 32 * tiny), ([2.0 ** -1022, -tiny], 2.0 ** -1022 - tiny),
                    ([big, big], np.inf), ([-big, -big], -np.inf), ([big, -big], 0.0), ([np.inf, 1.0], np.inf),
                    ([-np.inf, big], -np.inf), ([1.0, 2.0 ** -53], 1.0), ([1.0, 2.0 ** -53, 2.0 ** -76], 1 + 2.0 ** -52)):
        assert sum32(np.array(v)) == want, v
    for v in ([np.nan, 1.0], [np.inf, -np.inf], [np.nan, np.inf]):
        assert np.isnan(sum32(np.array(v)))


# Seven truncations below 2^-61 of the largest exponent's unit, one rounding.
@pytest.mark.parametrize("spread", [0, 2, 20, 59, 61, 64, 200, 1100])
def test_seven_terms(lib, spread):
    L, DP = lib
    rng = np.random.default_rng(spread)
    for k in range(500):
        v = np.ldexp(rng.uniform(1, 2, 7), rng.integers(-spread // 2, spread // 2 + 1, 7))
        v[rng.random(7) < 0.3] = 0.0
        v[k % 7] = max(v[k % 7], 2.0 ** -40)
        exact = sum(Fraction(float(x)) for x in v)
        top = Fraction(2) ** int(np.frexp(v.max())[1] - 1)
        assert abs(Fraction(L.ix_sum_seven(v.ctypes.data_as(DP))) - exact) <= exact / 2 ** 53 + 8 * top / 2 ** 61
    for bad in (-1.0, np.nan, np.inf, -0.0):
        v = np.ones(7)
        v[k % 7] = bad
        assert np.isnan(L.ix_sum_seven(v.ctypes.data_as(DP)))
    assert np.isnan(L.ix_sum_seven(np.zeros(7).ctypes.data_as(DP)))
