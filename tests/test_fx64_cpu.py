"""Fixed-point closures (csrc/fx64.cuh): the kernels' own source built for
the host, against the closed forms of Eq. 2-4 in 140-bit arithmetic, over the
soils and heads of the workloads and at the edges of its branches (x' = 2^-9,
m log2(1 + 1/x) = 2^-9, y = 0, the ends of its range)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1809_10895_gb300", "csrc")
DP = C.POINTER(C.c_double)


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    so = str(tmp_path_factory.mktemp("fx") / "libfx.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "c", "fx64_host.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.fx_init()
    L.fx_eval.argtypes = [C.c_double, C.c_double, DP, C.c_int, DP, DP, DP]

    def ev(alpha, n, h):
        h = np.ascontiguousarray(h)
        r = [np.empty(h.size) for _ in range(3)]
        L.fx_eval(alpha, n, h.ctypes.data_as(DP), h.size, *(a.ctypes.data_as(DP) for a in r))
        return r
    return ev


# Units of 2^-53.  y = n log2 u is carried to 2^-57 with an error of at most
# n 1.5 + 4 units of 2^-57 and a product by m adds 2, so Se's exponent is off
# by at most m (1.5 n + 4) + 2 <= 8 units (n <= 2.6) and Se by 8 ln2 / 16 <
# 0.35, plus its rounding (1).  K/Ks = Se^1/2 (1 - ys)^2: half of that, twice
# the relative error of 1 - ys (below 2 units wherever it is formed), its
# rounding: 6.  C/cfac: twice the exponent error and its rounding: 1.8.
TOL = {"se": 1.35, "k": 6.0, "c": 1.8}


@pytest.mark.parametrize("alpha,n", [(3.6, 1.56), (2.0, 1.8), (2.3, 1.2), (2.1, 2.4), (0.5, 1.25), (5.0, 2.6)])
def test_against_closed_forms(fx, alpha, n):
    mp.mp.prec = 140
    rng = np.random.default_rng(int(100 * alpha + 10 * n))
    m = float(1.0 - 1.0 / n)
    q9 = np.log2(1.0 / np.expm1(np.log(2.0) * 2.0 ** -9 / m))       # m log2(1 + 2^-y) = 2^-9
    edges = [y + d for y in (0.0, 9.0, -9.0, 8.0, -8.0, 10.0, -10.0, q9) for d in (-1e-3, -1e-9, 0.0, 1e-9, 1e-3)]
    h = np.concatenate([-10.0 ** rng.uniform(-6, 3, 60), -(2.0 ** (np.array(edges) / n)) / alpha,
                        -(2.0 ** (np.array([-31.0, -29.0, 29.0, 31.0, 59.9 / n, -59.9 / n]))) / alpha])
    se, k, c = fx(alpha, n, h)
    # all in range but the two heads beyond |log2 u| = 30
    assert np.isfinite(se).sum() >= h.size - 4
    for i in range(h.size):
        if not np.isfinite(se[i]):
            continue
        x = (-mp.mpf(alpha) * mp.mpf(float(h[i]))) ** mp.mpf(n)
        Se = (1 + x) ** -mp.mpf(m)
        omy = -mp.expm1(-mp.mpf(m) * mp.log1p(1 / x))
        for key, v, ref in (("se", se[i], Se), ("k", k[i], mp.sqrt(Se) * omy ** 2), ("c", c[i], (1 - omy) / (1 + x))):
            err = abs((mp.mpf(float(v)) - ref) / ref) * mp.mpf(2) ** 53
            assert err <= TOL[key], (key, alpha, n, h[i], float(err))


def test_out_of_range_heads_are_left_to_the_general_form(fx):
    h = np.array([-1e-300, -5e-324, -np.inf, -1e300, -2.0 ** 40, -2.0 ** -40])
    assert not np.isfinite(fx(2.0, 1.8, h)[0]).any()
