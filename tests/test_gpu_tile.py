"""The one-node-per-thread step (k_tile) where its choice of tile, its fast path and its dispatch can go wrong.

Oracle parity on edge sizes is held elsewhere (test_gpu_parity.py); here the step is compared with the
register-pipelined kernel (LBM_FLAG_NO_TMA), which shares the node update but neither the addressing nor the halo
handling, and with itself across the sizes at which a grid and its slabs take different kernels.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2111_00847_gb300 as pk

    return pk


def _state(pk, params, case, steps):
    with pk.Simulation(params) as s:
        s.init_fields(case.phi, case.ux, case.uy, case.p)
        s.step(steps)
        return [s.fields(w) for w in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST)]


# last strips and rows of one node, strips one node short of full, tiles that touch the periodic pads on both
# sides, blocks of every size (32 to 256 threads)
SIZES = [(4, 70), (17, 9), (33, 33), (65, 41), (993, 10), (130, 1027)]


@pytest.mark.parametrize("walls", ["none", "y", "x", "all"])
@pytest.mark.parametrize("model", [W.MODEL_AC, W.MODEL_CH])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_tile_step_matches_register_kernel(pk, nx, ny, model, walls):
    """One step differs by the rounding of a node update only (a few ulp of values of order one)."""
    for prec, tol in ((W.PREC_FP64, 1e-14), (W.PREC_FP32, 2e-6)):
        case = W.noisy_drop(nx, ny, precision=prec, model=model, walls=walls, noise=0.005, u_amp=0.002,
                            theta=(60, 120, 75, 105))
        tile = _state(pk, case.params, case, 1)
        march = _state(pk, case.params.with_(flags=pk.LBM_FLAG_NO_TMA), case, 1)
        for a, b in zip(tile[:2], march[:2]):
            assert np.abs(a - b).max() <= tol * np.abs(b).max()


@pytest.mark.parametrize("model", [W.MODEL_AC, W.MODEL_CH])
@pytest.mark.parametrize("prec", [W.PREC_FP16_DEV, W.PREC_FP32, W.PREC_FP64])
def test_slabs_across_the_dispatch(pk, prec, model):
    """A grid and its two slabs hold the same bits, with other tiles for the slabs (FP64: 16 x 4 against
    32 x 8) and other segments (16-bit)."""
    from paper_2111_00847_gb300 import slabs

    nx, ny = (500, 400) if prec == W.PREC_FP64 else (900, 700)
    case = W.noisy_drop(nx, ny, precision=prec, model=model, walls="y", noise=0.005, u_amp=0.002,
                        theta=(90, 90, 60, 120))
    whole = pk.Simulation(case.params)
    sims = [pk.Simulation(case.params, slab=band) for band in slabs.partition(ny, 2)]
    whole.init_fields(case.phi, case.ux, case.uy, case.p)
    for s in sims:
        s.init_fields(*(slabs.local_field(x, s) for x in (case.phi, case.ux, case.uy, case.p)))
    bufs = slabs.exchange_local(sims, periodic=False)
    for _ in range(4):
        whole.step(1)
        for s in sims:
            s.step(1)
        slabs.exchange_local(sims, periodic=False, bufs=bufs)
    for which in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST):
        ref = whole.fields(which)
        for s in sims:
            y_lo, own, glo, _ = s.slab
            assert np.array_equal(s.fields(which)[:, glo:glo + own], ref[:, y_lo:y_lo + own])
    for s in [whole, *sims]:
        s.close()


def test_small_n_delta_keeps_the_moment_form(pk):
    """FP64 with n_delta below its default, a channel under 16 columns: operation for operation the
    register kernel's update, so the same bits after many steps."""
    case = W.layered_poiseuille(nx=10, ny=100)
    a = _state(pk, case.params, case, 300)
    b = _state(pk, case.params.with_(flags=pk.LBM_FLAG_NO_TMA), case, 300)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
