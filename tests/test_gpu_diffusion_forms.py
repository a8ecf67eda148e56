"""The two launch forms of a diffusion call on 3D bodies: one tank is small enough for the
one-launch form, the same tank in a handle with copies of itself is not (the rule counts the
handle's particles) and runs as stage launches. Neighbours never cross tanks and a row's order
does not depend on the other tanks, so every copy's species equals the single tank's bit for bit."""
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


# 4 and 2 lanes a particle, one lane, and just above a lane each: two passes over the particles
@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("n, copies", [(33, 6), (42, 3), (50, 2), (54, 2)])
def test_one_launch_diffusion_equals_the_stage_launches_in_3d(sph, n, copies, masses):
    prob = wk.diffusion_block_3d(n)
    if masses:
        prob.mass = prob.mass * np.random.default_rng(1).uniform(0.9, 1.1, prob.mass.shape)
    C0 = np.random.default_rng(3).uniform(0.0, 1.0, prob.pos.shape[0])
    D = np.array([[2.0, 0.3, 0.1], [0.3, 1.0, 0.2], [0.1, 0.2, 0.5]]) if n == 50 else prob.meta["D"]
    out, launches = [], []
    for k in (1, copies):
        sim = sph.Simulation([prob] * k)
        sim.build_cells()
        sp = sph.sph_species_create(sim.handle, D, 3)
        sph.sph_species_set(sim.handle, sp, np.tile(C0, k))
        before = sim.kernel_launches()
        for _ in range(2):
            sph.sph_diffusion_step(sim.handle, sp, 0.3 * prob.meta["dt"], 2)
        launches.append(sim.kernel_launches() - before)
        out.append(sph.sph_species_get(sim.handle, sp, sim.n).reshape(k, -1))
        sph.sph_species_destroy(sp)
        sim.close()
    assert launches[0] == 2 < launches[1]            # a launch a call against several
    assert not np.array_equal(out[0][0], C0.astype(np.float32))
    for row in out[1]:
        np.testing.assert_array_equal(row, out[0][0])


@pytest.mark.parametrize("n", [550, 570])
def test_anisotropic_2d_calls_take_the_faster_form(sph, n):
    # up to two passes (2048 particles an SM) calls of a few steps run in one launch, past that
    # only those of one step; two calls of one step equal a call of two bit for bit
    per = -(-n * n // torch.cuda.get_device_properties(0).multi_processor_count)
    prob = wk.diffusion_band(n=n, ny=n)
    sim = sph.Simulation(prob)
    sim.build_cells()
    sp = sph.sph_species_create(sim.handle, np.array([[2.0, 0.3], [0.3, 1.0]]), 2)
    C0 = np.random.default_rng(3).uniform(0.0, 1.0, sim.n)
    out, launches = [], []
    for calls, steps in ((1, 2), (2, 1)):
        sph.sph_species_set(sim.handle, sp, C0)
        before = sim.kernel_launches()
        for _ in range(calls):
            sph.sph_diffusion_step(sim.handle, sp, 0.3 * prob.meta["dt"], steps)
        launches.append(sim.kernel_launches() - before)
        out.append(sph.sph_species_get(sim.handle, sp, sim.n))
    sph.sph_species_destroy(sp)
    sim.close()
    assert launches[1] == 2 and (launches[0] == 1) == (per <= 2048)
    np.testing.assert_array_equal(out[0], out[1])
