"""Array arguments of the wrappers: the library reads and writes plain doubles at the address it is given, so a tensor
that is no contiguous float64 one in reach is refused before the call."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")

SHAPE = (6, 5)
REFUSED = {
    "float32": lambda dev: torch.zeros(SHAPE, dtype=torch.float32, device=dev),
    "int64": lambda dev: torch.zeros(SHAPE, dtype=torch.int64, device=dev),
    "transposed": lambda dev: torch.zeros(SHAPE[::-1], dtype=torch.float64, device=dev).t(),
    "strided": lambda dev: torch.zeros((6, 10), dtype=torch.float64, device=dev)[:, ::2],
    "expanded": lambda dev: torch.zeros((1, 5), dtype=torch.float64, device=dev).expand(SHAPE),
    "sparse": lambda dev: torch.zeros(SHAPE, dtype=torch.float64, device=dev).to_sparse(),
}


@pytest.fixture
def pk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2111_00847_gb300 as pk

    return pk


def _dptr():
    from paper_2111_00847_gb300 import _dptr

    return _dptr


@pytest.mark.parametrize("name", sorted(REFUSED))
def test_host_tensors_of_another_form_are_refused(name):
    with pytest.raises(ValueError):
        _dptr()(REFUSED[name]("cpu"))


def test_tensors_elsewhere_are_refused():
    with pytest.raises(ValueError):
        _dptr()(torch.zeros(SHAPE, dtype=torch.float64, device="meta"))


def test_other_objects_are_refused():
    for a in ([1.0, 2.0], 3.0, "x"):
        with pytest.raises(AttributeError):
            _dptr()(a)


def test_host_arrays_and_tensors_give_their_address():
    a = np.zeros(SHAPE)
    t = torch.zeros(SHAPE, dtype=torch.float64)
    assert C.cast(_dptr()(a), C.c_void_p).value == a.ctypes.data
    assert C.cast(_dptr()(t), C.c_void_p).value == t.data_ptr()
    assert _dptr()(None) is None


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(REFUSED))
def test_device_tensors_of_another_form_are_refused(pk, name):
    case = W.noisy_drop(5, 6)
    with pk.Simulation(case.params) as s:
        bad = REFUSED[name]("cuda")
        for call in (lambda: pk.lbm_init_fields(s.handle, bad), lambda: pk.lbm_fields(s.handle, pk.LBM_PHI, bad),
                     lambda: pk.lbm_set_fields(s.handle, pk.LBM_HIST, bad), lambda: pk.lbm_adjoint_seed(s.handle, bad)):
            with pytest.raises(ValueError):
                call()
        with pytest.raises(ValueError):
            pk.lbm_adjoint_gravity(s.handle, torch.zeros(2, dtype=torch.float64, device="cuda"))


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
def test_device_arrays_hold_what_host_arrays_hold(pk, prec):
    """Fields, populations, history and a set state through device arrays: the same values."""
    case = W.noisy_drop(37, 29, precision=prec, walls="y", theta=(90, 90, 60, 120))
    dev = [torch.tensor(a, device="cuda") for a in (case.phi, case.ux, case.uy, case.p)]
    with pk.Simulation(case.params) as host, pk.Simulation(case.params) as s:
        host.init_fields(case.phi, case.ux, case.uy, case.p)
        pk.lbm_init_fields(s.handle, *dev)
        for sim in (host, s):
            sim.step(3)
        for which, n in ((pk.LBM_PHI, None), (pk.LBM_RHO, None), (pk.LBM_F_POP, 9), (pk.LBM_G_POP, 9), (pk.LBM_HIST, 5)):
            ref = host.fields(which)
            out = torch.full(ref.shape, 7.0, dtype=torch.float64, device="cuda")
            pk.lbm_fields(s.handle, which, out)
            assert np.array_equal(out.cpu().numpy(), ref)
            if n is not None:  # out of step by one, then set back
                s.step(1)
                for w in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST):
                    pk.lbm_set_fields(s.handle, w, torch.tensor(host.fields(w), device="cuda"))
        for w in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST):
            assert np.array_equal(s.fields(w), host.fields(w))


@pytest.mark.gpu
def test_diagnostics_into_a_device_array(pk):
    case = W.noisy_drop(37, 29)
    with pk.Simulation(case.params) as s:
        s.init_fields(case.phi, case.ux, case.uy, case.p)
        s.step(3)
        out = torch.full((pk.LBM_NDIAG,), 7.0, dtype=torch.float64, device="cuda")
        pk.lbm_fields(s.handle, pk.LBM_DIAG, out)
        assert np.array_equal(out.cpu().numpy(), s.fields(pk.LBM_DIAG))
