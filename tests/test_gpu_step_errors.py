"""sph_step on small single tanks (one cooperative launch a step, or one for all steps of a call
with SPH_FLAG_PERSISTENT) stops at the first step that fails: what it leaves is what a call of
exactly the steps up to that one leaves, in every loop mode, and the handle goes on from a new
state. The launches of a call are enqueued before the first status is read, so the later ones
have to find the failure themselves."""
import numpy as np
import pytest

from paper_2010_12375_gb300 import workloads as wk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_12375_gb300 import sph as s
    s.load()
    return s


MODES = ["host", "graph", "persistent"]


def _flags(sph, mode):
    return {"host": 0, "graph": sph.SPH_FLAG_GRAPH, "persistent": sph.SPH_FLAG_PERSISTENT}[mode]


def _left(sph, sim, steps, code):
    """What a failing call of `steps` steps leaves."""
    with pytest.raises(sph.SphError) as e:
        sim.step(steps)
    assert e.value.code == code
    sph.sph_clear_error(sim.handle)
    d = sim.diagnostics()
    return [*sim.state(), sim.permutation(), np.array([d["advection_steps"], d["substeps"], d["t"], d["dt_ad"]])]


def _case(sph, fault):
    """A tank whose first step fails: the problem, the handle's options, its start and the code."""
    prob = wk.dam_break_2d(n_per_H=20)
    x = prob.pos.copy()
    if fault == "domain":
        x[5, 0] = prob.hi[0] + 1.0
    opt = {"bound": {"max_substeps": 1}, "capacity": {"capacity": 8}, "domain": {}}[fault]
    code = {"bound": sph.SPH_E_TIMEOUT, "capacity": sph.SPH_E_CAPACITY, "domain": sph.SPH_E_DOMAIN}[fault]
    return prob, opt, x, code


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("fault", ["bound", "capacity", "domain"])
def test_a_call_stops_at_a_failing_first_step(sph, fault, mode):
    prob, opt, x, code = _case(sph, fault)
    out = []
    for steps in (1, 4):
        sim = sph.Simulation(prob, flags=_flags(sph, mode), **opt)
        sim.set_state(x, prob.vel, prob.rho, t=0.0)
        out.append(_left(sph, sim, steps, code))
        if fault == "domain":                        # and on from a good state, as a new handle
            sim.set_state(prob.pos, prob.vel, prob.rho, t=0.0)
            sim.step(3)
            new = sph.Simulation(prob, flags=_flags(sph, mode))
            new.step(3)
            for a, b in zip(sim.state(), new.state()):
                np.testing.assert_array_equal(a, b)
            new.close()
        sim.close()
    assert out[0][-1][0] == 1
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_a_call_stops_at_a_failing_later_step(sph):
    # a particle flies off a free sheet and leaves the grid some steps into the call: every loop
    # mode ends with the step whose hash finds it
    prob = wk.excitable_sheet(12)
    v = prob.vel.copy()
    v[-1] = (4.0, 0.0)
    out = []
    for mode in MODES:
        sim = sph.Simulation(prob, flags=_flags(sph, mode))
        sim.set_state(prob.pos, v, prob.rho, t=0.0)
        out.append(_left(sph, sim, 60, sph.SPH_E_DOMAIN))
        sim.close()
    k = int(out[0][-1][0])
    assert 1 < k < 60
    sim = sph.Simulation(prob)                       # the steps before it pass
    sim.set_state(prob.pos, v, prob.rho, t=0.0)
    sim.step(k - 1)
    sim.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b)
