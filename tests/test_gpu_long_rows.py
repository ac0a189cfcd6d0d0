"""Rows longer than 2^20 elements, which a tile's 32-bit offsets do not reach, run on the register-pipelined kernel, the
one-thread-per-node pass (obstacles) and the general adjoint.  A field that repeats along x must give there what one
period of it gives on the tile kernels."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NX, REP, NY = 1056, 1024, 3  # 1,081,344 columns


@pytest.fixture(scope="module")
def pk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2111_00847_gb300 as pk

    return pk


def _rep(a):
    return np.tile(a, (1, REP))


@pytest.mark.parametrize("model,prec,solid", [(W.MODEL_AC, W.PREC_FP32, False), (W.MODEL_AC, W.PREC_FP64, False),
                                              (W.MODEL_CH, W.PREC_FP32, False), (W.MODEL_CH, W.PREC_FP64, False),
                                              (W.MODEL_AC, W.PREC_FP32, True), (W.MODEL_AC, W.PREC_FP64, True)])
def test_step_on_long_rows(pk, model, prec, solid):
    """One step, the rounding of a node update apart (a few ulp of values of order one)."""
    case = W.noisy_drop(NX, NY, precision=prec, model=model, noise=0.005, u_amp=0.002)
    m = np.zeros((NY, NX), bool)
    m[1, 300:303] = m[2, 0] = True
    tol = 1e-14 if prec == W.PREC_FP64 else 2e-6
    with pk.Simulation(case.params) as one, pk.Simulation(case.params.with_(nx=NX * REP)) as all_:
        for s, rep in ((one, lambda a: a), (all_, _rep)):
            if solid:
                s.set_solid(rep(m))
            s.init_fields(*(rep(a) for a in (case.phi, case.ux, case.uy, case.p)))
            s.step(1)
        for which in (pk.LBM_F_POP, pk.LBM_G_POP):
            a = one.fields(which)
            b = all_.fields(which).reshape(9, NY, REP, NX)
            assert np.abs(b - a[:, :, None, :]).max() <= tol * np.abs(a).max()


def test_gradient_on_long_rows(pk):
    from paper_2111_00847_gb300.adjoint import rollout

    case = W.noisy_drop(NX, NY, noise=0.005, gravity=(W.GRAV_RHO, 1e-5, -2e-5))
    wts = W.uniform_array(7, NX * NY).reshape(NY, NX) - 0.5
    out = []
    for rep, prm in ((lambda a: a, case.params), (_rep, case.params.with_(nx=NX * REP))):
        phi0 = torch.tensor(rep(case.phi), requires_grad=True)
        G = torch.tensor([prm.gx, prm.gy], dtype=torch.float64, requires_grad=True)
        (rollout(phi0, G, prm, 3, 2) * torch.from_numpy(rep(wts))).sum().backward()
        out.append((phi0.grad.numpy(), G.grad.numpy()))
    (p1, g1), (p2, g2) = out
    assert np.abs(p2.reshape(NY, REP, NX) - p1[:, None, :]).max() <= 1e-9 * np.abs(p1).max()
    assert np.abs(g2 / REP - g1).max() <= 1e-9 * np.abs(g1).max()
