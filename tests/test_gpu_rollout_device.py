"""rollout with phi0 on the device: the same numbers as with phi0 on the host, for strided and FP32 leaves."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _grads(torch, rollout, case, device, dtype, strided):
    phi = torch.tensor(case.phi, dtype=dtype, device=device)
    if strided:
        phi = phi.t().contiguous().t()
    phi.requires_grad_(True)
    G = torch.tensor([case.params.gx, case.params.gy], dtype=dtype, device=device, requires_grad=True)
    phi_n = rollout(phi, G, case.params, 7, 3)
    w = torch.from_numpy(W.uniform_array(5, phi_n.numel()).reshape(phi_n.shape)).to(device)
    (phi_n * w).sum().backward()
    return [t.detach().cpu() for t in (phi_n, phi.grad, G.grad)]


@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("nx,ny", [(40, 33), (257, 65)])
def test_device_leaf_matches_host_leaf(nx, ny, prec, strided):
    torch = pytest.importorskip("torch")
    from paper_2111_00847_gb300.adjoint import rollout

    case = W.noisy_drop(nx, ny, precision=prec, walls="y", theta=(90, 90, 60, 120),
                        gravity=(W.GRAV_RHO_MINUS_MEAN, 0.0, -2e-5))
    dtype = torch.float64 if prec == W.PREC_FP64 else torch.float32
    for a, b in zip(*(_grads(torch, rollout, case, d, dtype, strided) for d in ("cuda", "cpu"))):
        assert torch.equal(a, b)


def test_device_leaf_of_another_shape_is_refused():
    torch = pytest.importorskip("torch")
    from paper_2111_00847_gb300.adjoint import rollout

    case = W.noisy_drop(40, 33, precision=W.PREC_FP64)
    G = torch.zeros(2, dtype=torch.float64)
    with pytest.raises(ValueError):
        rollout(torch.tensor(case.phi, device="cuda").t(), G, case.params, 2, 1)
