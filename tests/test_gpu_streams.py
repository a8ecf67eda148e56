"""Handles of their own on streams and host threads of their own, stepped at the same time: the
cooperative launches of one (a step or a diffusion call of a small tank, the persistent substeps
of several tanks) beside the other's give the results of each run alone."""
import threading

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


def _jobs(sph):
    def step(prob, flags):
        def run(stream):
            sim = sph.Simulation(prob, flags=flags, stream=stream)
            for _ in range(10):
                sim.step(3)
            out = sim.state()
            sim.close()
            return out
        return run

    def diffuse(prob):
        def run(stream):
            sim = sph.Simulation(prob, stream=stream)
            sim.build_cells()
            sp = sph.sph_species_create(sim.handle, prob.meta["D"], prob.dim)
            sph.sph_species_set(sim.handle, sp, prob.meta["C0"], stream=stream)
            for _ in range(50):
                sph.sph_diffusion_step(sim.handle, sp, prob.meta["dt"], 1, stream=stream)
            out = (sph.sph_species_get(sim.handle, sp, sim.n, stream=stream),)
            sph.sph_species_destroy(sp)
            sim.close()
            return out
        return run

    return [step(wk.dam_break_2d(n_per_H=100), sph.SPH_FLAG_GRAPH), step(wk.dam_break_3d(20), 0),
            diffuse(wk.diffusion_patch(200)),
            step([wk.dam_break_2d(n_per_H=n) for n in (40, 60, 80)], sph.SPH_FLAG_PERSISTENT)]


def test_handles_on_streams_of_their_own_run_side_by_side(sph):
    jobs = _jobs(sph)
    alone = [job(None) for job in jobs]
    streams = [torch.cuda.Stream() for _ in jobs]
    got = [None] * len(jobs)

    def work(k):
        got[k] = jobs[k](streams[k].cuda_stream)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, got):
        assert b is not None
        for u, v in zip(a, b):
            np.testing.assert_array_equal(u, v)
