"""Fixed-point closures of soils with n near 1, where m and 1 - ys are small
at every head: the kernels' own source built for the host with the library's
soil constants, against 200-bit arithmetic."""
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
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    so = str(tmp_path_factory.mktemp("fx") / "libfxs.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "c", "fx64_soil_host.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.fx_init()
    L.fx_takes_soil.argtypes = [C.c_double, C.c_double]
    L.fx_eval.argtypes = [C.c_double, C.c_double, DP, C.c_int, DP, DP, DP]
    return L


# Units of 2^-53, as for larger n.  K: 1 - ys is at least 2^-9.5 where it is
# formed from 2^-q in Q64, with six units of Q64 from the power and q (2.2
# units of 2^-53), and relative below; twice that and one rounding and half of
# Se's exponent error make 6.
TOL = {"se": 1.35, "k": 6.0, "c": 1.8}


@pytest.mark.parametrize("n", [1.07, 1.066, 1.05, 1.02, 1.01, 1.005, 1.002, 1.001, 1.0005, 1.0003, 1.000245])
def test_n_near_one(lib, n):
    mp.mp.prec = 200
    alpha = 2.0
    rng = np.random.default_rng(int(1e6 * n))
    m = float(1.0 - 1.0 / n)
    edges = [0.0, 9.0, -9.0]
    for q in (2.0 ** -9, 1.0):                # q = m log2(1 + 1/x) at its branches, where some head reaches it
        b = q / m * np.log(2.0)
        edges.append(-b / np.log(2.0) if b > 30 else np.log2(1.0 / np.expm1(b)))
    edges = np.array([y + d for y in edges if abs(y) < 28 for d in (-1e-3, -1e-9, 0.0, 1e-9, 1e-3)])
    h = np.concatenate([-10.0 ** rng.uniform(-6, 3, 80), -(2.0 ** rng.uniform(-29, 29, 80)) / alpha,
                        -(2.0 ** rng.uniform(-1, 1, 40)) / alpha, -(2.0 ** (edges / n)) / alpha])
    r = [np.empty(h.size) for _ in range(3)]
    lib.fx_eval(alpha, n, h.ctypes.data_as(DP), h.size, *(a.ctypes.data_as(DP) for a in r))
    assert np.isfinite(r[0]).all()
    for i in range(h.size):
        x = (-mp.mpf(alpha) * mp.mpf(float(h[i]))) ** mp.mpf(n)
        Se = (1 + x) ** -mp.mpf(m)
        omy = -mp.expm1(-mp.mpf(m) * mp.log1p(1 / x))
        for (key, tol), v, ref in zip(TOL.items(), (a[i] for a in r), (Se, mp.sqrt(Se) * omy ** 2, (1 - omy) / (1 + x))):
            err = abs((mp.mpf(float(v)) - ref) / ref) * mp.mpf(2) ** 53
            assert err <= tol, (key, n, h[i], float(err))


def test_soils_left_to_the_general_form(lib):
    # m below 2^-12 is not exact in Q64
    assert not any(lib.fx_takes_soil(2.0, n) for n in (1.0001, 1.000001, 16.0, 20.0))
    assert all(lib.fx_takes_soil(2.0, n) for n in (1.000245, 1.2, 15.9))
