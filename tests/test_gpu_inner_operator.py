"""The FP32 inner stencil step against the oracle's operator, element by
element, in the form that each route's iterations run: the sweep of the
one-launch solve also where nx is a multiple of 4, and the TMA-staged kernel of
the loops (multigrid, DIC, Jacobi without one-launch solves)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from tests import test_gpu_parity as P
from tests.helpers import oracle_from_case
from tests.test_gpu_parity import gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("precond,solves", [("jacobi", True), ("jacobi", False), ("dic", True)])
@pytest.mark.parametrize("make", [P._box_multitile, P._watershed_multitile, P._box_wide, P._box_odd])
def test_matches_oracle(make, precond, solves):
    case = make()
    o = oracle_from_case(case)
    s = rf.Solver.from_case(case, precision="mixed", precond=precond)
    s.set_one_launch(solves=solves)
    rng = np.random.default_rng(31)
    hk = case.h0 + rng.normal(0, 0.02, case.N)
    s.assemble(gpu(hk), gpu(case.h0), 90.0, 0.0)
    mask = np.ones(case.N, bool) if case.active is None else case.active.astype(bool)
    act = o.active_cells
    z, pold = (torch.as_tensor(rng.standard_normal(case.N), dtype=torch.float32, device="cuda") for _ in range(2))
    for beta in (0.0, 0.37):
        p, q = torch.zeros_like(z), torch.zeros_like(z)
        pq = s.apply_inner(z, p, q, pold=pold, beta=beta)
        pg, qg = p.cpu().numpy().astype(np.float64), q.cpu().numpy().astype(np.float64)
        # one rounding of z + beta p_old, 0 off the active set
        pr = z.cpu().numpy().astype(np.float64) + float(np.float32(beta)) * pold.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(pg - pr)[mask] <= 2.0 ** -24 * np.abs(pr[mask]) + 2.0 ** -50)
        assert np.all(pg[~mask] == 0) and np.all(qg[~mask] == 0)
        qo = o.spmv(hk, case.h0, 90.0, pg[act])
        assert np.all(np.abs(qg[act] - qo) <= P._inner_operator_bound(case, o, hk, case.h0, 90.0, pg, act))
        assert pq == pytest.approx(float(pg[act] @ qo), rel=1e-5)
