"""The one-launch Picard attempt of small grids against the oracle: one block
and several, grids around the switch between them, masks, every time scheme
and Picard form, and a second context beside the first."""
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


def _check(s, o, case, n, tol):
    for _ in range(n):
        a, b = s.step(), o.step()
        assert (a.dt, a.picard, a.rejected) == (b.dt, b.picard, b.rejected)
    hg, ho = s.get_state()[0], o.get_state()[0]
    act = np.ones(case.N, bool) if case.active is None else case.active.astype(bool)
    assert np.max(np.abs(hg - ho)[act]) <= tol
    mg, mo = s.mass_balance(), o.mass_balance()
    for k in ("storage", "inflow_cum", "outflow_cum"):
        assert abs(mg[k] - mo[k]) <= 1e-9 * (mo["storage0"] + abs(mo[k]))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(1, 1, 8), (1, 1, 512), (8, 8, 8), (9, 19, 3), (19, 3, 11), (40, 33, 25)])
def test_steps_match_oracle(shape, precision):
    case = W.heterogeneous_box(*shape, d=0.25, seed=sum(shape), water_table_depth=1.5, rain=5e-6, tol_cg=1e-13,
                               dt0=60.0)
    _check(rf.Solver.from_case(case, precision=precision), oracle_from_case(case), case, 6, TOL[precision])


@pytest.mark.parametrize("over", [dict(picard_form="modified"), dict(picard_form="modified", time_scheme="bdf2"),
                                  dict(grav=(0.2, 0.0, 0.95))])
@pytest.mark.parametrize("shape", [(7, 5, 12), (20, 13, 12)])
def test_options_match_oracle(shape, over):
    case = W.watershed(*shape, dx=2.0, dz=0.5, seed=5, tol_cg=1e-13, dt0=400.0)      # masked columns
    case.bcs[0] = W.BC("zmax", "flux", np.array([0.0]), np.array([2e-6]))
    if "grav" in over:
        case.gravity = over["grav"]
    opt = {k: v for k, v in over.items() if k != "grav"}
    o = oracle_from_case(case, **{k: 1 for k in opt})
    _check(rf.Solver.from_case(case, **opt), o, case, 8, TOL["fp64"])


def test_two_contexts_on_two_streams():
    case = W.heterogeneous_box(20, 13, 12, d=0.25, seed=7, water_table_depth=1.5, rain=5e-6, tol_cg=1e-13)
    with torch.cuda.stream(torch.cuda.Stream()):
        a = rf.Solver.from_case(case)
    with torch.cuda.stream(torch.cuda.Stream()):
        b = rf.Solver.from_case(case)
    for _ in range(4):
        ia, ib = a.step(), b.step()
        assert (ia.dt, ia.picard, ia.cg) == (ib.dt, ib.picard, ib.cg)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
