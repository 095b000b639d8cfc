"""Closures of the mixed path's automatic arithmetic: fixed point (bit for bit
the FP64 choice's) inside its range, double-float (bit for bit that choice's)
outside it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("alpha,n,inside", [(2.0, 1.8, (-1e3, -1e-6)), (14.0, 7.0, (-20.0, -0.01)), (4.0, 20.0, None),
                                            (2.0, 1.0001, None)])
def test_auto_on_the_mixed_path(alpha, n, inside):
    rng = np.random.default_rng(int(10 * n))
    h = -10.0 ** rng.uniform(-14, 3, 2000)
    if inside is None:
        ins = np.zeros(h.size, bool)
    else:
        L = np.abs(np.log2(-alpha * h))
        ins, out = (L < 29.5) & (n * L < 59.5), (L > 31.5) | (n * L > 60.5)
        h, ins = h[ins | out], ins[ins | out]
        assert ins.any() and not ins.all()
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    got = {}
    for arith in ("auto", "fp64", "double_float"):
        s = rf.Solver(1, 1, h.size, 1.0, 1.0, 0.1, 0.0,
                      params=rf.default_params(precision="mixed", closure_arith=arith))
        s.set_soils([dict(theta_r=0.05, theta_s=0.40, alpha=alpha, n=n, Ks=1e-5, S=1e-5)])
        K, th = dev(np.zeros(h.size)), dev(np.zeros(h.size))
        s.assemble(dev(h), dev(h - 0.25), 10.0, 0.0, K=K, theta=th)
        got[arith] = np.stack([K.cpu().numpy(), th.cpu().numpy()])
    assert np.array_equal(got["auto"], np.where(ins, got["fp64"], got["double_float"]))
    assert not np.array_equal(got["fp64"], got["double_float"])
