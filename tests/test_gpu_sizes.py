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
