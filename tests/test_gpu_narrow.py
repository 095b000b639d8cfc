"""Solves and steps of grids whose planes leave their tiles mostly empty
(columns, vertical sections), which run cell by cell, and of grids on the other
side of that line, against the oracle: masks and every boundary type, one-launch
solves, loops and DIC; heads that are not numbers on masked cells."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from paper_1809_10895_gb300 import workloads as W
from tests.helpers import oracle_from_case
from tests.test_gpu_parity import gpu, masked_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


# 8 x 15 of a 32 x 16 tile is below a quarter, 8 x 16 is not
@pytest.mark.parametrize("shape", [(1, 1, 700), (1, 40, 9), (40, 1, 9), (5, 3, 50), (8, 15, 7), (8, 16, 7)])
@pytest.mark.parametrize("precision,precond,solves", [("fp64", "jacobi", True), ("fp64", "jacobi", False),
                                                      ("mixed", "jacobi", True), ("mixed", "jacobi", False),
                                                      ("mixed", "dic", True)])
def test_solve_matches_oracle(shape, precision, precond, solves):
    case = masked_case(*shape, seed=sum(shape))
    o, s = oracle_from_case(case), rf.Solver.from_case(case, precision=precision, precond=precond)
    s.set_one_launch(solves=solves)
    hk = case.h0 + np.random.default_rng(3).normal(0, 0.02, case.N)
    s.assemble(gpu(hk), gpu(case.h0), 120.0, 0.0)
    x = gpu(hk)
    assert s.solve(x) > 0
    act = o.active_cells
    # both residuals are at most 1e-13 |b|; heads of order 1 m, condition below 1e4
    assert np.max(np.abs(x.cpu().numpy()[act] - o.solve(hk, case.h0, 120.0)[0])) <= 1e-8


@pytest.mark.parametrize("precision,precond,solves", [("fp64", "jacobi", True), ("mixed", "jacobi", True),
                                                      ("mixed", "jacobi", False), ("mixed", "dic", True)])
def test_masked_section_steps(precision, precond, solves):
    case = W.watershed(40, 2, 24, dx=2.0, dz=32.0 / 24, seed=5, tol_cg=1e-13, dt0=200.0)
    case.bcs[0] = W.BC("zmax", "flux", np.array([0.0]), np.array([2e-6]))
    act = np.asarray(case.active, bool)
    assert not act.all()
    o = oracle_from_case(case)
    ho = [o.step() for _ in range(3)]
    for fill in (0.0, np.nan):
        s = rf.Solver.from_case(case, precision=precision, precond=precond)
        s.set_one_launch(attempts=False, solves=solves)
        s.set_state_device(gpu(np.where(act, case.h0, fill)), 0.0)
        got = [s.step() for _ in range(3)]
        assert [(i.dt, i.picard, i.rejected) for i in got] == [(i.dt, i.picard, i.rejected) for i in ho]
        assert np.max(np.abs(s.get_state()[0] - o.get_state()[0])[act]) <= (1e-8 if precision == "fp64" else 1e-6)
