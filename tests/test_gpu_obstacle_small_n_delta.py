"""FP64 Allen-Cahn runs with n_delta below its default keep the node update's moment form with obstacles as they do
without: started from the same state, nodes that an obstacle has not reached yet hold the bits of the run without it."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

NX, NY = 256, 96


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2111_00847_gb300 as pk

    return pk


def _pair(pk, prm, case, steps):
    """Fields without and with an obstacle, set after the initial state (whose kernels may round otherwise), and the
    columns it has not reached: a node reaches at most 3 nodes a step (a pull, and the stencil of phi)."""
    solid = np.zeros((NY, NX), bool)
    solid[40:46, 118:126] = True
    out = []
    for m in (None, solid):
        with pk.Simulation(prm) as s:
            s.init_fields(case.phi, case.ux, case.uy, case.p)
            s.set_solid(m)
            s.step(steps)
            out.append([s.fields(w) for w in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST)])
    return out, np.abs(np.arange(NX) - 121.5) > 4.5 + 3 * steps


@pytest.mark.parametrize("s_g", [None, (1.0, 1.1, 0.9, 1.0, 1.7, 1.0, 1.7, float("nan"), float("nan"))],
                         ids=["unit_rates", "other_rates"])
@pytest.mark.parametrize("walls", ["none", "y"])
@pytest.mark.parametrize("nd", [1e-5, 3e-3])
def test_tile_step_far_from_the_obstacle(pk, nd, walls, s_g):
    case = W.noisy_drop(NX, NY, walls=walls, noise=0.005, u_amp=0.002, theta=(90, 90, 60, 120), s_g=s_g)
    (plain, obs), far = _pair(pk, case.params.with_(n_delta=nd), case, 12)
    for a, b in zip(plain, obs):
        assert np.array_equal(a[:, :, far], b[:, :, far])


@pytest.mark.parametrize("nd", [1e-5, 3e-3])
def test_node_pass_far_from_the_obstacle(pk, nd):
    """The one-thread-per-node pass beside the register-pipelined kernel: the compiler fuses the collisions of two
    kernels differently, the history (phi u, u.m) comes out the same."""
    case = W.noisy_drop(NX, NY, walls="y", noise=0.005, u_amp=0.002, theta=(90, 90, 60, 120))
    (plain, obs), far = _pair(pk, case.params.with_(n_delta=nd, flags=pk.LBM_FLAG_NO_TMA), case, 1)
    assert np.array_equal(plain[2][:, :, far], obs[2][:, :, far])
