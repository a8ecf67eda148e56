"""The launch-per-phase loops of single tanks (host, CUDA graph, persistent substeps) and the
launch forms of the relaxations in them, on tanks larger than sph_step runs in one launch a step.
Each run asserts by its launch counter that it did not take that form: smaller tanks would, and a
comparison of two of these loops on them would compare the one-launch step with itself."""
import numpy as np
import pytest

from paper_2010_12375_gb300 import workloads as wk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEPS = 2


@pytest.fixture(scope="module")
def sph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_12375_gb300 import sph as s
    s.load()
    return s


def _tank(case):
    """The least sizes past the one-launch limits (704 particles an SM in 2D, 192 in 3D)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if case == "dam3d":
        n = next(n for n in range(8, 99) if 2 * n ** 3 > 192 * sms)
        return wk.dam_break_3d(n)
    if case == "dam2d":
        n = next(n for n in range(8, 999) if 2 * n ** 2 > 704 * sms)
        return wk.dam_break_2d(n_per_H=n)
    n = next(n for n in range(8, 999) if n ** 2 > 704 * sms)
    return wk.taylor_green(n=n, transport=True)


def _run(sph, prob, flags, cfg=None, steps=STEPS):
    """State and clock after `steps` steps; the launches are those of separate phases."""
    sim = sph.Simulation(prob, flags=flags)
    if cfg is not None:
        sph.sph_set_launch_config(sim.handle, cfg)
    x = prob.pos + np.random.default_rng(2).uniform(-0.05, 0.05, prob.pos.shape) * prob.dp
    if np.any(prob.periodic[:prob.dim]):
        x = np.mod(x, 1.0)
    sim.set_state(x, prob.vel, prob.rho, t=0.0)
    before = sim.kernel_launches()
    sim.step(steps)
    assert sim.kernel_launches() - before > 5 * steps
    d = sim.diagnostics()
    out = [*sim.state(), np.array([d["substeps"], d["advection_steps"], d["t"], d["dt_ad"]])]
    sim.close()
    return out


def _same(a, b):
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("case", ["dam3d", "dam2d", "tg_tv"])
def test_loops_agree_bit_for_bit(sph, case):
    prob = _tank(case)
    host, graph, pers = (_run(sph, prob, f) for f in (0, sph.SPH_FLAG_GRAPH, sph.SPH_FLAG_PERSISTENT))
    assert host[-1][0] > STEPS                       # several substeps a step
    _same(host, graph)
    _same(host, pers)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("case", ["dam3d", "dam2d", "tg_tv"])
def test_launch_forms_agree_bit_for_bit(sph, case, graph):
    # one, two and four threads a particle and the row tasks, alone and mixed
    prob = _tank(case)
    flags = sph.SPH_FLAG_GRAPH if graph else 0
    ref = _run(sph, prob, flags, [1, 128, 1, 128])
    for cfg in ([1, 896, 1, 896], [1, 896, 1, 256], [4, 128, 2, 512]):
        _same(ref, _run(sph, prob, flags, cfg))


def test_graph_stops_at_the_substep_bound(sph):
    prob = _tank("dam3d")
    sim = sph.Simulation(prob, flags=sph.SPH_FLAG_GRAPH, max_substeps=1)
    before = sim.kernel_launches()
    for k in (1, 2):
        with pytest.raises(sph.SphError) as e:
            sim.step(1)
        assert e.value.code == sph.SPH_E_TIMEOUT
        sph.sph_clear_error(sim.handle)
        d = sim.diagnostics()
        assert d["substeps"] == k and d["advection_steps"] == k
    assert sim.kernel_launches() - before > 10
    assert all(np.all(np.isfinite(a)) for a in sim.state())
    sim.close()


def test_graph_takes_a_new_gravity(sph):
    prob = _tank("dam3d")
    a = sph.Simulation(prob, flags=sph.SPH_FLAG_GRAPH)
    a.step(1)
    x, v, rho, drho = a.state()
    t = a.diagnostics()["t"]
    g = np.array([0.3, -0.8, 0.1])
    sph.sph_set_gravity(a.handle, g)
    before = a.kernel_launches()
    a.step(2)
    assert a.kernel_launches() - before > 10
    other = _tank("dam3d")
    other.gravity = g.copy()
    b = sph.Simulation(other)
    b.set_state(x, v, rho, drho, t=t)
    b.step(2)
    _same(a.state(), b.state())
    a.close()
    b.close()
