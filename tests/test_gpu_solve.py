"""The one-launch CG solves (FP64, and FP32 inside FP64 defect correction) on
grids around their tiles' sizes against the oracle's solve, and heads that are
not numbers on masked cells in every path of a step."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(1, 1, 5), (33, 17, 7), (31, 16, 40), (64, 32, 3), (130, 33, 9), (5, 70, 2)])
def test_solve_matches_oracle(shape, precision):
    case = masked_case(*shape, seed=sum(shape))
    o, s = oracle_from_case(case), rf.Solver.from_case(case, precision=precision)
    rng = np.random.default_rng(3)
    hk = case.h0 + rng.normal(0, 0.02, case.N)
    s.assemble(gpu(hk), gpu(case.h0), 120.0, 0.0)
    x = gpu(hk)
    it = s.solve(x)
    act = o.active_cells
    ref, _, _ = o.solve(hk, case.h0, 120.0)
    assert it > 0 or len(act) <= 1
    # both residuals are at most 1e-13 |b|; heads of order 1 m, condition below 1e4
    assert np.max(np.abs(x.cpu().numpy()[act] - ref)) <= 1e-8


@pytest.mark.parametrize("precision,precond", [("fp64", "jacobi"), ("mixed", "jacobi"), ("mixed", "dic")])
@pytest.mark.parametrize("shape", [(20, 13, 12), (96, 96, 64)])
def test_masked_cells_may_hold_anything(shape, precision, precond):
    case = W.watershed(*shape, dx=2.0, dz=32.0 / shape[2], seed=5, dt0=200.0)
    case.bcs[0] = W.BC("zmax", "flux", np.array([0.0]), np.array([2e-6]))
    act = np.asarray(case.active, bool)
    assert not act.all()
    heads = []
    for fill in (0.0, np.nan):
        s = rf.Solver.from_case(case, precision=precision, precond=precond)
        s.set_state_device(gpu(np.where(act, case.h0, fill)), 0.0)
        infos = [s.step() for _ in range(2)]
        heads.append((s.get_state()[0][act], [(i.picard, i.cg, i.rejected) for i in infos]))
    assert heads[0][1] == heads[1][1]
    assert np.array_equal(heads[0][0], heads[1][0])


@pytest.mark.parametrize("shape,precision", [((96, 96, 64), "fp64"), ((96, 96, 64), "mixed"), ((40, 40, 30), "fp64")])
def test_contexts_step_in_parallel_threads(shape, precision):
    """Each launch's blocks wait for one another only; two contexts' launches
    may be on the GPU at once."""
    import threading
    case = W.heterogeneous_box(*shape, d=0.25, seed=2, water_table_depth=4.0, rain=2e-6, dt0=30.0)

    def run(out, k):
        torch.cuda.set_device(0)
        with torch.cuda.stream(torch.cuda.Stream()):
            s = rf.Solver.from_case(case, precision=precision)
            infos = [s.step() for _ in range(4)]
            out[k] = (s.get_state()[0], [(i.dt, i.picard, i.cg) for i in infos])

    alone, both = {}, {}
    run(alone, 0)
    ts = [threading.Thread(target=run, args=(both, k)) for k in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for k in range(3):
        assert both[k][1] == alone[0][1]
        assert np.array_equal(both[k][0], alone[0][0])
