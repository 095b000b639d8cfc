"""Bounded device waits that run out: the call returns RF_ERR_DEVICE_TIMEOUT
with the state unchanged, and the context then steps as if nothing had been."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf, warmstart
from paper_1809_10895_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


def _box():
    return W.heterogeneous_box(20, 13, 12, d=0.25, seed=7, water_table_depth=1.5, rain=5e-6, dt0=60.0, f_grow=1.0)


def _network():
    net = rf.Network()
    net.set_params(W.nn_init_params(6))
    return net


def _times_out(s):
    h0, m0 = s.get_state()
    s.set_wait_limit(-1)
    with pytest.raises(rf.RFError) as e:
        s.step()
    assert e.value.status == rf.RF_ERR_DEVICE_TIMEOUT
    s.set_wait_limit(0)
    h1, m1 = s.get_state()
    assert np.array_equal(h0, h1) and m0 == m1


def _same_steps(a, b, n):
    for _ in range(n):
        i, j = a.step(), b.step()
        assert (i.dt, i.picard, i.cg, i.rejected, i.max_dh) == (j.dt, j.picard, j.cg, j.rejected, j.max_dh)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])


def test_network_guess():
    """A wait of the network's convolutions; then warm-started steps again."""
    case, net = _box(), _network()
    sc = warmstart.scales_for(case, out_scale=1e-6)
    s, ref = rf.Solver.from_case(case), rf.Solver.from_case(case)
    for c in (s, ref):
        c.ws_attach(net, sc)
        c.step()
    _times_out(s)
    _same_steps(s, ref, 3)


def test_plain_step_after_a_guess_that_timed_out():
    """The closures of the guess (here metres off, left in the network's
    output by the step before) do not pass for the state's."""
    case, net = _box(), _network()
    sc = warmstart.scales_for(case, out_scale=5.0 / 60.0)
    s, ref = rf.Solver.from_case(case), rf.Solver.from_case(case)
    for c in (s, ref):
        c.ws_attach(net, sc)
        c.step()
    _times_out(s)
    for c in (s, ref):
        c.ws_attach(None)
    _same_steps(s, ref, 3)
