"""Kernels at the sizes where their splits can go wrong (tile edges, remainders, the smallest
and largest of a launch rule's range), against the oracle or the library's general path."""
import numpy as np
import pytest

from oracle import mpnn
from oracle import wcsph as o
from paper_2010_12375_gb300 import workloads as wk
from tests.parity import perturbed_state, rel_l2, representable, walls_representable

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_12375_gb300 import sph as s
    s.load()
    return s


def _block(nx, ny, dp=0.02):
    """nx x ny fluid particles at rest in a tank corner, on the library's grid."""
    prob = wk.dam_break(dim=2, H=ny * dp, L=nx * dp, dp=dp, tank=max(nx, ny, 12) * dp + 0.2)
    prob.wall_pos = walls_representable(prob)
    return prob


@pytest.mark.parametrize("nx, ny", [(1, 1), (8, 8), (13, 5), (70, 45)])
def test_weight_gradients_at_tile_edges(sph, nx, ny):
    # the weight gradients split the node and edge rows in 64-row tiles over blocks: one row,
    # one whole tile, one row over, and edge rows spread over every block with several tiles each
    prob = _block(nx, ny)
    st = representable(prob, *perturbed_state(prob, 3, 0.3, 0.01))
    W = mpnn.init_weights(2, seed=9)
    flat = np.concatenate([W[k].ravel() for k in ("enc", "e1", "e2", "n1", "n2", "d1", "d2")]).astype(np.float32)
    net = sph.sph_learned_create(2, flat)
    sim = sph.Simulation(prob)
    sim.set_state(*st, t=0.0)
    sim.build_cells()
    dt_ad = sim.advection_step()
    pos, vel, rho, _ = sim.state()
    T = np.random.default_rng(4).normal(0.0, 0.5, size=(prob.n_fluid, 3))
    _, grad = sph.sph_learned_train_step(sim.handle, net, T, 0.0, want_grad=True)
    prm = o.Params.from_problem(prob)
    I, J, IW, KW = o.neighbour_sets_quantised(pos, prob.wall_pos, prm)
    g = mpnn.build_graph(2, pos, vel, rho, prob.wall_pos, I, J, IW, KW, prob.h, prob.c0, prob.rho0, dt_ad)
    W32 = {k: v.astype(np.float32).astype(np.float64) for k, v in W.items()}
    Y, cache = mpnn.forward(W32, g)
    dW = mpnn.backward(W32, g, cache, Y, T)
    at = 0
    for k in ("enc", "e1", "e2", "n1", "n2", "d1", "d2"):
        got = grad[at:at + dW[k].size].reshape(dW[k].shape)
        at += dW[k].size
        if np.linalg.norm(dW[k]) > 0:
            assert rel_l2(got, dW[k]) < 1e-3, k        # the bound the weight gradients are held to
    sph.sph_learned_destroy(net)
    sim.close()


def _fused_case(name):
    """Tanks that sph_step runs in one launch a step, at the lane counts' edges (8, 4, 2, 1
    lanes a particle by the particles an SM holds) and with each of the step's options."""
    if name.startswith("2d"):
        nx, ny = {"2d_one": (1, 1), "2d_three": (3, 1), "2d_9728": (128, 76), "2d_9729": (423, 23),
                  "2d_19456": (152, 128), "2d_30600": (180, 170), "2d_visc": (37, 29)}[name]
        prob = wk.dam_break(dim=2, H=ny * 0.02, L=nx * 0.02, dp=0.02, tank=max(nx, ny, 12) * 0.02 + 0.3)
        if name == "2d_visc":
            prob.nu = 0.01
    elif name.startswith("tg"):
        prob = wk.taylor_green({"tg_48": 48, "tg_230": 230}[name])
    elif name == "box3d":
        prob = wk.periodic_box(dim=3, n=12, seed=2)
    else:
        prob = wk.dam_break_3d({"3d_11": 11, "3d_17": 17, "3d_24": 24}[name])
        prob.nu = 0.002 if name == "3d_17" else 0.0
    if name in ("2d_three", "3d_11"):                # masses that differ: a per-particle array
        prob.mass = prob.mass * np.random.default_rng(3).uniform(0.95, 1.05, prob.mass.shape)
    return prob


@pytest.mark.parametrize("case", ["2d_one", "2d_three", "2d_9728", "2d_9729", "2d_19456", "2d_30600", "2d_visc",
                                  "tg_48", "tg_230", "box3d", "3d_11", "3d_17", "3d_24"])
def test_one_launch_step_equals_the_per_launch_loop(sph, case):
    # every sum of the one-launch step adds the same terms in the same order: state, table,
    # acceleration, clock and substep count agree bit for bit (kernel timing keeps sph_step on
    # the per-launch kernels), in the host, graph and all-steps-in-one-launch forms
    prob = _fused_case(case)
    rng = np.random.default_rng(7)
    x = prob.pos + rng.uniform(-0.1, 0.1, prob.pos.shape) * prob.dp
    v = prob.vel + rng.uniform(-0.2, 0.2, prob.vel.shape)
    if np.any(prob.periodic[:prob.dim]):
        x = np.mod(x, 1.0)
    out = []
    for flags, timing in ((0, True), (0, False), (sph.SPH_FLAG_GRAPH, False), (sph.SPH_FLAG_PERSISTENT, False)):
        sim = sph.Simulation(prob, flags=flags | sph.SPH_FLAG_KEEP_ACC)
        sim.set_state(x, v, prob.rho, t=0.0)
        sph.sph_set_kernel_timing(sim.handle, timing)
        before = sim.kernel_launches()
        sim.step(3)
        launches = sim.kernel_launches() - before
        assert launches > 20 if timing else launches == (1 if flags == sph.SPH_FLAG_PERSISTENT else 3)
        d = sim.diagnostics()
        fc, wc, fi, wi = sim.neighbours()
        rows = [np.concatenate([fi[i, :fc[i]], wi[i, :wc[i]]]) for i in range(0, sim.n, max(1, sim.n // 500))]
        out.append((*sim.state(), sim.acceleration(), sim.permutation(), fc, wc, np.concatenate(rows),
                    np.array([d["substeps"], d["t"], d["dt_ad"], d["advection_steps"]])))
        sim.step(1)                                  # and on from there
        out[-1] = out[-1] + sim.state()
        sim.close()
    for o_ in out[1:]:
        for a, b in zip(out[0], o_):
            np.testing.assert_array_equal(a, b)


def test_one_launch_step_reports_errors_and_goes_on(sph):
    # a row beyond the capacity and a particle outside the grid: the codes of the other loops,
    # and the handle steps on after a new state
    prob = wk.dam_break_2d(n_per_H=20)
    sim = sph.Simulation(prob, capacity=8)
    with pytest.raises(sph.SphError) as e:
        sim.step(2)
    assert e.value.code == sph.SPH_E_CAPACITY
    sim.close()
    ref, sim = sph.Simulation(prob), sph.Simulation(prob)
    x = prob.pos.copy()
    x[5, 0] = prob.hi[0] + 1.0
    sim.set_state(x, prob.vel, prob.rho, t=0.0)
    with pytest.raises(sph.SphError) as e:
        sim.step(2)
    assert e.value.code == sph.SPH_E_DOMAIN
    sph.sph_clear_error(sim.handle)
    for s in (ref, sim):
        s.set_state(prob.pos, prob.vel, prob.rho, t=0.0)
        s.step(3)
    for a, b in zip(ref.state(), sim.state()):
        np.testing.assert_array_equal(a, b)
    ref.close()
    sim.close()


@pytest.mark.parametrize("case", ["3d_11", "2d_visc"])
def test_threads_per_particle_change_no_bit(sph, case):
    # the lanes of a particle add its terms in row order (kernel timing: per-launch kernels)
    prob = _fused_case(case)
    out = []
    for cfg in ([1, 128, 1, 128], [2, 128, 4, 256], [4, 512, 2, 512]):
        sim = sph.Simulation(prob)
        sph.sph_set_launch_config(sim.handle, cfg)
        sph.sph_set_kernel_timing(sim.handle, True)
        sim.step(3)
        out.append(sim.state())
        sim.close()
    for o_ in out[1:]:
        for a, b in zip(out[0], o_):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("case", ["sheet", "sheet_masses", "box2d_aniso", "block3d", "block3d_scale"])
def test_one_launch_diffusion_equals_the_stage_launches(sph, case):
    # above one lane a particle a call of five steps runs as stage launches and a call of one
    # step as one launch: five of the latter give the same bits
    D = None
    if case.startswith("sheet"):
        prob = wk.diffusion_patch(400)
    elif case == "box2d_aniso":
        prob, D = wk.diffusion_band(n=400, ny=400), np.array([[2.0, 0.3], [0.3, 1.0]])
    else:
        prob = wk.diffusion_block_3d(55)
    if case == "sheet_masses":
        prob.mass = prob.mass * np.random.default_rng(1).uniform(0.9, 1.1, prob.mass.shape)
    sim = sph.Simulation(prob)
    sim.build_cells()
    sp = sph.sph_species_create(sim.handle, prob.meta["D"] if D is None else D, prob.dim)
    if case.endswith("scale"):
        sph.sph_species_set_scale(sim.handle, sp, np.random.default_rng(2).uniform(0.5, 2.0, sim.n))
    C0 = np.random.default_rng(3).uniform(0.0, 1.0, sim.n)
    out = []
    for calls, steps in ((1, 5), (5, 1)):
        sph.sph_species_set(sim.handle, sp, C0)
        l0 = sim.kernel_launches()
        for _ in range(calls):
            sph.sph_diffusion_step(sim.handle, sp, 0.5 * prob.meta["dt"], steps)
        assert sim.kernel_launches() - l0 == (12 if calls == 1 else 5)
        out.append(sph.sph_species_get(sim.handle, sp, sim.n))
    np.testing.assert_array_equal(out[0], out[1])
    assert not np.array_equal(out[0], C0.astype(np.float32))
    sph.sph_species_destroy(sp)
    sim.close()


@pytest.mark.parametrize("nx, ny", [(3, 1), (4, 33), (130, 75), (131, 75), (220, 190), (480, 330)])
def test_fused_edge_rounds_at_run_boundaries(sph, nx, ny):
    # node runs of the shortest length (and one node past it), of a whole tile of nodes and
    # two more, and several runs a warp; tiles of edges with every remainder: the same bits as
    # the layers one by one
    prob = _block(nx, ny)
    sim = sph.Simulation(prob)
    sim.build_cells()
    sim.advection_step()
    W = mpnn.init_weights(2, seed=6)
    net = sph.sph_learned_create(2, np.concatenate([W[k].ravel() for k in ("enc", "e1", "e2", "n1", "n2", "d1", "d2")]))
    y = []
    for form in (1, 0):
        sph.sph_learned_set_fused(net, form)
        y.append(sph.sph_learned_predict(sim.handle, net, prob.n_fluid, 2))
    assert np.all(np.isfinite(y[0])) and np.abs(y[0]).max() > 0
    np.testing.assert_array_equal(y[0], y[1])
    sph.sph_learned_destroy(net)
    sim.close()


# solid steps in registers: one block, a short last block, every block full and 16 blocks
@pytest.mark.parametrize("ratio, L, thickness", [(1, 0.2, 0.1), (2, 0.2, 0.05), (4, 0.3, 0.0375), (4, 0.2, 0.05),
                                                 (4, 0.825, 0.05625)])
def test_solid_steps_over_the_blocks_of_a_cluster(sph, ratio, L, thickness):
    from tests.test_gpu_fsi import _coupled_substep_against_oracle, _prepared
    wl, prm = _prepared(ratio, wl=wk.water_column_on_plate(dp=1.0 / 40.0, ratio=ratio, H=0.2, L=L, thickness=thickness))
    _coupled_substep_against_oracle(sph, wl, prm, f"ratio {ratio} L {L} thickness {thickness}")
