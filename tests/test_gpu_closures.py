"""Closures on the GPU at the edges of the fixed-point form: heads inside,
at and beyond its range, soils that it does not take, masked cells and grids
around a block's size, against the oracle's closures (K of van Genuchten
soils against Eq. 4 with 1 - ys = -expm1(-m log1p(1/x)): the oracle's literal
1 - Se^(1/m) has no digits left within 1e-6 m of saturation)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1809_10895_gb300 import rf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


SOILS = [dict(theta_r=0.05, theta_s=0.40, alpha=2.0, n=1.8, Ks=1e-5, S=1e-5),
         dict(theta_r=0.08, theta_s=0.45, alpha=2.3, n=1.2, Ks=1e-3, S=1e-5),
         dict(theta_r=0.10, theta_s=0.35, alpha=4.0, n=20.0, Ks=1e-4, S=1e-4),     # n too large for it
         dict(theta_r=0.05, theta_s=0.40, alpha=1.5, n=1.0, Ks=1e-6, S=1e-5, model="gardner")]


@pytest.mark.parametrize("nz", [1, 31, 255, 257, 2000])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_edges_of_the_range(nz, precision):
    rng = np.random.default_rng(nz)
    zone = rng.integers(0, len(SOILS), nz).astype(np.uint8)
    active = (rng.random(nz) < 0.9).astype(np.uint8)
    active[0] = 1
    pool = np.concatenate([-10.0 ** rng.uniform(-6, 3, 40), -2.0 ** np.array([-31.5, -30.5, -29.5, 28.5, 30.5, 45.0]),
                           [-1e-12, -1e-200, 0.0, -0.0, 1.5, -1.0, -0.5]])
    h = rng.choice(pool, nz)
    s = rf.Solver(1, 1, nz, 1.0, 1.0, 0.1, 0.0, active, params=rf.default_params(precision=precision,
                                                                                   closure_arith="fp64"))
    s.set_soils(SOILS, zone)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    K, th = dev(np.zeros(nz)), dev(np.zeros(nz))
    s.assemble(dev(h), dev(h - 0.25), 10.0, 0.0, K=K, theta=th)
    K, th = K.cpu().numpy(), th.cpu().numpy()
    for p in range(nz):
        if not active[p]:
            assert K[p] == -1.0 and th[p] == 0.0
            continue
        soil = SOILS[zone[p]]
        rt, rk, _ = O.closure(dict(soil, model=O.GARDNER if soil.get("model") else O.VG), float(h[p]))
        if not soil.get("model") and h[p] < 0.0:
            m, lx = 1.0 - 1.0 / soil["n"], soil["n"] * math.log(-soil["alpha"] * h[p])
            l1 = lx + math.log1p(math.exp(-lx)) if lx > 0 else math.log1p(math.exp(lx))        # log(1 + x)
            rk = soil["Ks"] * math.exp(-0.5 * m * l1) * math.expm1(m * (lx - l1 if lx < 30 else -math.exp(-lx))) ** 2
        # theta: the oracle's pow form and this one each within 1e-15; K: a
        # few thousand units of the last place in m log(x/(1+x))
        assert abs(th[p] - rt) <= 2e-15 * abs(rt), (p, soil, h[p])
        if np.isfinite(rk):
            assert abs(K[p] - rk) <= 2e-11 * abs(rk) + 1e-15 * soil["Ks"], (p, soil, h[p])
