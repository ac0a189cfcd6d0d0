"""Which snapshots one kernel may copy (pflbm_copy.h, compiled for the host): only a buffer that holds the state, in
16-byte words, in memory of the handle's device, while that device is current.  Every other buffer goes to copy
commands, which find both devices themselves and refuse a range that its allocation does not hold."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_00847_gb300", "csrc")

SOURCE = r"""
#include "pflbm_copy.h"
extern "C" int by_kernel(uint64_t addr, int device_memory, int device, uint64_t start, uint64_t size, uint64_t parts,
                         long long bytes, int handle_device, int current_device) {
  return pflbm::copy_by_kernel({(uintptr_t)addr, device_memory != 0, device, (uintptr_t)start, size}, (uintptr_t)parts,
                               bytes, handle_device, current_device);
}
"""

OK = dict(addr=0x7f0000000000, device_memory=1, device=0, start=0x7f0000000000, size=1 << 21, parts=0x7e0000000100,
          bytes=1 << 20, handle_device=0, current_device=0)


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("copy")
    src, so = d / "copy.cpp", d / "copy.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True)
    fn = C.CDLL(str(so)).by_kernel
    fn.argtypes = [C.c_uint64, C.c_int, C.c_int, C.c_uint64, C.c_uint64, C.c_uint64, C.c_longlong, C.c_int, C.c_int]
    return lambda **kw: fn(*{**OK, **kw}.values())


@pytest.mark.parametrize("kw", [
    {}, dict(bytes=1 << 21), dict(addr=OK["addr"] + (1 << 20)), dict(device=3, handle_device=3, current_device=3),
])
def test_the_kernel_takes(rule, kw):
    assert rule(**kw) == 1


@pytest.mark.parametrize("kw", [
    dict(current_device=1),                             # it would run on the wrong GPU
    dict(device=1), dict(device=1, current_device=1),   # the buffer lies on another GPU
    dict(device_memory=0),
    dict(addr=OK["addr"] + 8), dict(parts=OK["parts"] + 8),
    dict(bytes=(64 << 20) + 16, size=1 << 30),
    dict(bytes=(1 << 21) + 16), dict(addr=OK["addr"] + (1 << 20) + 16), dict(size=0), dict(size=(1 << 20) - 16),
    dict(addr=OK["addr"] - 16), dict(addr=OK["addr"] + (1 << 22)),
])
def test_the_copies_take(rule, kw):
    assert rule(**kw) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 8, 16])
def test_snapshots_at_any_offset_restore_the_same_state(offset):
    import numpy as np

    import workloads as W

    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2111_00847_gb300 as pk

    case = W.noisy_drop(61, 47, precision=W.PREC_FP32)
    with pk.Simulation(case.params) as s:
        s.init_fields(case.phi, case.ux, case.uy, case.p)
        s.step(3)
        buf = torch.full((s.state_bytes + 64,), 7, dtype=torch.uint8, device="cuda")
        s.snapshot(buf[offset:])
        whole = s.snapshot(s.new_state_buffer())
        assert torch.equal(buf[offset:offset + s.state_bytes], whole)
        assert bool((buf[:offset] == 7).all()) and bool((buf[offset + s.state_bytes:] == 7).all())
        ref = [s.fields(w) for w in (pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST)]
        s.step(4)
        s.restore(buf[offset:], 3)
        for w, a in zip((pk.LBM_F_POP, pk.LBM_G_POP, pk.LBM_HIST), ref):
            assert np.array_equal(s.fields(w), a)
