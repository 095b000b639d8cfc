"""The tiled assembly (grids of at least 32768 cells) against the oracle:
ragged tiles, masked columns, every boundary type, tilted gravity, both Picard
forms, the harmonic mean, cells on and off the chord branch.  (Steps on it:
the 132 x 24 x 16 watershed and the full-size box in test_gpu_parity.py.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from tests.helpers import oracle_from_case
from tests.test_gpu_parity import chord_tol, gpu, masked_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("shape", [(37, 29, 33), (33, 9, 128), (16, 64, 33), (130, 5, 67), (64, 32, 16)])
@pytest.mark.parametrize("form", ["chord", "modified", "tilted", "harmonic"])
def test_tiled_assembly_matches_oracle(shape, form):
    case = masked_case(*shape, seed=sum(shape))
    over = {"chord": {}, "modified": dict(picard_form="modified"), "tilted": {}, "harmonic": dict(face_mean="harmonic")}
    if form == "tilted":
        case.gravity = (0.3, 0.1, 0.9)
    o = oracle_from_case(case, **{k: 1 for k in over[form]})
    s = rf.Solver.from_case(case, **over[form])
    rng = np.random.default_rng(9)
    hk = case.h0 + rng.normal(0, 0.05, case.N) * (rng.random(case.N) < 0.8)      # a fifth on the tangent branch
    out = {k: torch.zeros(case.N, dtype=torch.float64, device="cuda") for k in ("K", "theta", "c", "b", "diag")}
    s.assemble(gpu(hk), gpu(case.h0), 37.0, 0.0, **out)
    ref = o.assemble(hk, case.h0, 37.0, 0.0)
    act = o.active_cells
    got = {k: v.cpu().numpy()[act] for k, v in out.items()}
    tol_c = chord_tol(case, hk, case.h0, 37.0, act, ref["c"])
    tol_c = np.where(np.abs(hk - case.h0)[act] > 0, tol_c, 2e-12 * np.abs(ref["c"]))
    assert np.all(np.abs(got["c"] - ref["c"]) <= tol_c)
    assert np.all(np.abs(got["diag"] - ref["diag"]) <= tol_c + 2e-12 * ref["diag"])
    # b = c h^n (or c h^k - V dtheta/dt: theta's own 1e-15 of V/dt) + gravity + boundary terms
    V_dt = case.dx * case.dy * case.dz / 37.0
    tol_b = tol_c * np.maximum(np.abs(case.h0), np.abs(hk))[act] + 2e-15 * V_dt + 1e-11 * np.abs(ref["b"]) \
        + 1e-14 * np.abs(ref["b"]).max()
    assert np.all(np.abs(got["b"] - ref["b"]) <= tol_b)
    # the face coefficients, through the operator
    x = rng.normal(0, 1.0, case.N)
    y = torch.zeros(case.N, dtype=torch.float64, device="cuda")
    s.apply(gpu(x), y)
    yr = o.spmv(hk, case.h0, 37.0, x[act])
    assert np.all(np.abs(y.cpu().numpy()[act] - yr) <= tol_c * np.abs(x[act]) + 1e-11 * ref["diag"] * 4.0)

