"""Steps on the route of large grids (tiled assembly, one-launch solves inside
the Picard graph) and on the loops it falls back to, against the oracle at
sizes that would take the small-grid attempt: ragged tiles, masks, every
Picard form, time scheme and control, tilted gravity, both precisions; and
contexts on a stream that is limited to a few SMs."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from paper_1809_10895_gb300 import workloads as W
from tests.helpers import oracle_from_case

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-8, "mixed": 1e-6}      # m, as in the parity tests


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


# 45 x 29 and 45 x 30 fill 0.64 and 0.66 of their assembly tiles: tiled, ragged
# (harmonic mean: one cell per thread)
def _box(shape=(45, 29, 33), **k):
    return W.heterogeneous_box(*shape, d=0.25, seed=9, water_table_depth=2.0, rain=5e-6, tol_cg=1e-13, dt0=60.0, **k)


def _watershed(**k):
    c = W.watershed(45, 30, 32, dx=2.0, dz=1.0, seed=5, tol_cg=1e-13, dt0=200.0, **k)      # a sixth of the cells masked
    c.bcs[0] = W.BC("zmax", "flux", np.array([0.0]), np.array([2e-6]))
    return c


def _slope(**k):
    return W.tilted_slope(nx=45, ny=29, nz=32, days=0.25, tol_cg=1e-13, dt0=120.0, **k)


CASES = {"box": (_box, {}), "masked": (_watershed, {}), "tilted": (_slope, {}),
         "modified": (_watershed, dict(picard_form=1)), "tilted_modified": (_slope, dict(picard_form=1)),
         "bdf2": (_watershed, dict(picard_form=1, time_scheme=1)), "harmonic": (_box, dict(face_mean=1)),
         "harmonic_tiled": (_box, dict(face_mean=1, shape=(95, 24, 16))),
         "richardson": (_box, dict(time_control=1, tol_time=2e-3))}


@pytest.mark.parametrize("solves", [True, False], ids=["one_launch", "loops"])
@pytest.mark.parametrize("precision,name", [(p, n) for p in ("fp64", "mixed") for n in CASES
                                            if p == "fp64" or "harmonic" not in n])
def test_steps_match_oracle(name, precision, solves):
    make, over = CASES[name]
    case = make(**over)
    s, o = rf.Solver.from_case(case, precision=precision), oracle_from_case(case)
    s.set_one_launch(attempts=False, solves=solves)
    before = s.launch_counts()
    for _ in range(4):
        a, b = s.step(), o.step()
        # Richardson's dt is a continuous function of the solutions' difference
        assert a.dt == pytest.approx(b.dt, rel=1e-5 if name == "richardson" else 0, abs=0)
        assert (a.picard, a.rejected) == (b.picard, b.rejected)
    act = np.ones(case.N, bool) if case.active is None else case.active.astype(bool)
    assert np.max(np.abs(s.get_state()[0] - o.get_state()[0])[act]) <= TOL[precision]
    mg, mo = s.mass_balance(), o.mass_balance()
    for k in ("storage", "inflow_cum", "outflow_cum"):
        assert abs(mg[k] - mo[k]) <= 1e-9 * (mo["storage0"] + abs(mo[k]))
    n = {k: v[1] - before[k][1] for k, v in s.launch_counts().items()}
    assert n["closure_picard"] > 0 and (n["one_launch"] > 0) == solves
    assert (n["cg64_update"] + n["cg32_update"] > 0) == (not solves)


@pytest.fixture(scope="module")
def green(tmp_path_factory):
    """A stream of 16 SMs."""
    if not shutil.which("gcc"):
        pytest.skip("no gcc")
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("green") / "libgreen.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    os.path.join(here, "c", "green_stream.c"), "-o", so], check=True)
    C.CDLL("libcuda.so.1", mode=C.RTLD_GLOBAL)
    lib, ctx, stream = C.CDLL(so), C.c_void_p(), C.c_void_p()
    torch.zeros(1, device="cuda")
    assert lib.green_stream(0, 16, C.byref(ctx), C.byref(stream)) == 0
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    lib.green_free.argtypes = [C.c_void_p, C.c_void_p]
    assert lib.green_free(ctx, stream) == 0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(40, 33, 25), (96, 96, 64)])
def test_stream_of_few_sms(green, shape, precision):
    """More blocks than the stream's SMs hold: the context takes the launches
    of a graph instead of failing."""
    case = W.heterogeneous_box(*shape, d=0.25, seed=2, water_table_depth=4.0, rain=2e-6, dt0=30.0, tol_cg=1e-13)
    ref = rf.Solver.from_case(case, precision=precision)
    with torch.cuda.stream(green):
        s = rf.Solver.from_case(case, precision=precision)
        for _ in range(3):
            a, b = s.step(), ref.step()
            assert (a.dt, a.picard, a.rejected) == (b.dt, b.picard, b.rejected)
        h = s.get_state()[0]
        x = torch.as_tensor(case.h0, dtype=torch.float64, device="cuda")
        s.assemble(x, x, 30.0, 0.0)
        assert s.solve(x.clone()) > 0
        s.close()
    assert np.max(np.abs(h - ref.get_state()[0])) <= TOL[precision]
