"""Grids whose tiles are no multiple of a warp (7 x 4 threads, 5 x 51, 3 x 42): the Cahn-Hilliard step and the compact
adjoint fill the whole halo ring of such tiles.  Between the runs' set-up and their steps another simulation leaves
values of 5 in the shared memory, so that a cell nobody stores cannot hold the right one by chance."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2111_00847_gb300 as pk

    return pk


def _stain(pk, prec, model):
    case = W.noisy_drop(700, 600, precision=prec, model=model)
    with pk.Simulation(case.params) as s:
        s.init_fields(np.full((600, 700), 5.0))
        s.step(2)


@pytest.mark.parametrize("prec,nx,ny", [(W.PREC_FP64, n, n) for n in (14, 33, 42, 49)] + [(W.PREC_FP64, 14, 28)] +
                         [(W.PREC_FP32, n, 200) for n in (3, 5, 6, 7, 9)])
def test_ch_step_on_tiles_of_partial_warps(pk, prec, nx, ny):
    """Against the register-pipelined kernel after 1 and 20 steps: a node update's rounding, and the parity bar."""
    case = W.noisy_drop(nx, ny, precision=prec, model=W.MODEL_CH, noise=0.005, u_amp=0.002,
                        gravity=(W.GRAV_RHO, 1e-6, -1e-5))
    sims = [pk.Simulation(case.params.with_(flags=fl)) for fl in (0, pk.LBM_FLAG_NO_TMA)]
    for s in sims:
        s.init_fields(case.phi, case.ux, case.uy, case.p)
    fp64 = prec == W.PREC_FP64
    for steps, tol in ((1, 1e-14 if fp64 else 2e-6), (19, 1e-12 if fp64 else 1e-5)):
        for s in sims:
            _stain(pk, prec, W.MODEL_CH)
            s.step(steps)
        for which in (pk.LBM_F_POP, pk.LBM_G_POP):
            a, b = (s.fields(which) for s in sims)
            assert np.abs(a - b).max() <= tol * np.abs(b).max()
    for s in sims:
        s.close()


@pytest.mark.parametrize("nx,ny", [(3, 100), (3, 300), (31, 40)])
def test_adjoint_on_tiles_of_partial_warps(pk, nx, ny):
    """FP32 gradients (32 x 4, here 3 x 42 and 31 x 4 threads) against FP64 ones (other tiles).  FP32 rounds phi to
    6e-8, which turns the normal, of slope up to 1 / delta_n = 800 per unit of gradient, by 5e-5; over the 6 + 6 steps
    1e-3 of the largest component leaves room for twenty such errors in a row."""
    from paper_2111_00847_gb300.adjoint import rollout

    out = []
    for prec in (W.PREC_FP64, W.PREC_FP32):
        case = W.noisy_drop(nx, ny, precision=prec, walls="none", noise=0.005, gravity=(W.GRAV_RHO, 1e-5, -2e-5))
        wts = torch.from_numpy(W.uniform_array(7, nx * ny).reshape(ny, nx) - 0.5)
        phi0 = torch.tensor(case.phi, requires_grad=True)
        G = torch.tensor([case.params.gx, case.params.gy], dtype=torch.float64, requires_grad=True)
        phi_n = rollout(phi0, G, case.params, 6, 3)
        _stain(pk, prec, W.MODEL_AC)
        (phi_n * wts).sum().backward()
        out.append([t.detach().numpy() for t in (phi_n, phi0.grad, G.grad)])
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-3 * np.abs(a).max()


@pytest.mark.parametrize("nx,ny", [(3, 40), (7, 30), (29, 400)])
def test_gravity_gradient_on_blocks_of_partial_warps(pk, nx, ny):
    """dJ/dG sums over blocks of 30, 28 and 60 threads; the bar of the adjoint's other comparisons with autograd."""
    from oracle.torch_ref import TorchScheme
    from paper_2111_00847_gb300.adjoint import rollout

    case = W.noisy_drop(nx, ny, walls="y", noise=0.01, gravity=(W.GRAV_RHO, 1e-5, -2e-5))
    wts = torch.from_numpy(W.uniform_array(7, nx * ny).reshape(ny, nx) - 0.5)
    grads = []
    for run in (lambda phi, G: TorchScheme(case.params).run(phi, G, 8)[0], lambda phi, G: rollout(phi, G, case.params, 8, 3)):
        phi0 = torch.tensor(case.phi, requires_grad=True)
        G = torch.tensor([case.params.gx, case.params.gy], dtype=torch.float64, requires_grad=True)
        (run(phi0, G) * wts).sum().backward()
        grads.append((phi0.grad, G.grad))
    for a, b in zip(*grads):
        assert (a - b).abs().max() <= 1e-9 * a.abs().max()
