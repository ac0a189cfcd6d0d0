"""recip and inv_root4 (FP64), on which every FP64 node update rests, against extended precision.

Bounds, in units of 2^-53 relative, from the series (pflbm_kernels.cuh), with the hardware seeds good to 2^-19.9 (1 / a)
and 2^-19.7 (S^-1/4):
  recip      1 (the last rounding) + 2 e (the roundings of e and of e + e^2) + e^3 / 2^-53 = 0.011, e = 2^-19.9: 1.02;
  inv_root4  1 + 3 / 4 (the rounding of z^2, twice, and of S z^2, in e, of which a quarter enters)
             + 15/128 e^3 / 2^-53 = 0.11, e = 4 * 2^-19.7: 1.9.
Range: densities and viscous denominators (far inside 1e-8 .. 1e8); |grad phi|^4 + delta^4 from its floor 1e-290 up."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "pflbm_kernels.cuh"
__global__ void k(const double* a, double* r, double* q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = pflbm::recip(a[i]), q[i] = pflbm::inv_root4(a[i]);
}
extern "C" int run(const double* a, double* r, double* q, int n) {
  k<<<(n + 255) / 256, 256>>>(a, r, q, n);
  const cudaError_t e = cudaGetLastError();
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_00847_gb300 import build as b

    d = tmp_path_factory.mktemp("seeds")
    src, so = d / "seeds.cu", d / "seeds.so"
    src.write_text(SOURCE)
    subprocess.run([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared",
                    "-I", b.CSRC, str(src), "-o", str(so)], check=True)
    lib = C.CDLL(str(so))

    def run(x):
        a = torch.tensor(x, device="cuda")
        r, q = torch.empty_like(a), torch.empty_like(a)
        torch.cuda.synchronize()
        assert lib.run(C.c_void_p(a.data_ptr()), C.c_void_p(r.data_ptr()), C.c_void_p(q.data_ptr()), x.size) == 0
        return r.cpu().numpy(), q.cpu().numpy()

    return run


def _mantissas():
    """All seeds' table entries (2^21 equal steps of [1, 4)), each at a random place inside its step."""
    rng = np.random.default_rng(1)
    n = 1 << 21
    return 1.0 + 3.0 * (np.arange(n) + rng.random(n)) / n


def _worst(got, exact):
    return float((np.abs(got.astype(np.longdouble) - exact) / np.abs(exact)).max() * np.longdouble(2) ** 53)


@pytest.mark.parametrize("scale", [1e-8, 0.25, 1.0, 1e8])
def test_recip(evaluate, scale):
    a = _mantissas() * scale
    assert _worst(evaluate(a)[0], 1 / a.astype(np.longdouble)) <= 1.02
    assert _worst(evaluate(-a)[0], -1 / a.astype(np.longdouble)) <= 1.02


@pytest.mark.parametrize("scale", [1e-290, 1e-200, 4e-17, 2e-11, 1.0, 4.0, 1e6])
def test_inv_root4(evaluate, scale):
    a = np.concatenate([[1e-290], np.maximum(_mantissas() * scale, 1e-290)])
    assert _worst(evaluate(a)[1], 1 / np.sqrt(np.sqrt(a.astype(np.longdouble)))) <= 1.9
