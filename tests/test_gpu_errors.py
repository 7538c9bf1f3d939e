"""Calls after a call that failed (GPU)."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402
from paper_2204_03775_gb300 import binding  # noqa: E402

SHAPE = (12, 40, 80)


def _handle():
    nz, ny, nx = SHAPE
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_set_velocity(h, np.full(SHAPE, 3000.0, np.float32))
    return h


def _cudart():
    """The CUDA runtime that the library itself is linked to."""
    binding.load_library()
    with open("/proc/self/maps") as f:
        paths = {line.split()[-1] for line in f if "libcudart.so" in line}
    libs = [ctypes.CDLL(p) for p in sorted(paths)]
    assert libs
    return libs


@pytest.mark.parametrize("where", ["library", "caller"])
@pytest.mark.parametrize("call", ["write", "write_zero", "read", "velocity", "step", "energy", "storage"])
def test_a_failed_allocation_fails_no_later_call(where, call):
    """The error of an allocation that failed, in an earlier call or in the
    caller's own code, is not taken for one of the next call's launches."""
    h = _handle()
    u, out = (torch.rand(SHAPE, device="cuda") for _ in range(2))
    v = torch.full(SHAPE, 3000.0, device="cuda")
    wsb.ws_write_field(h, u, u, 0)
    wsb.ws_step(h, 1)
    wsb.ws_synchronize(h)
    if where == "library":
        with pytest.raises(wsb.WaveStepError) as e:      # 550 GB of traces
            wsb.ws_set_receivers(h, np.zeros((64, 3), np.int32), 2 ** 31 - 1)
        assert e.value.code == wsb.WS_ERR_OOM
    else:
        for lib in _cudart():
            p = ctypes.c_void_p()
            assert lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(1 << 45)) != 0
    if call == "write":
        wsb.ws_write_field(h, u, u, 0)
    elif call == "write_zero":
        wsb.ws_write_field(h, None, None, 0)
    elif call == "read":
        wsb.ws_read_field(h, out, None)
    elif call == "velocity":
        wsb.ws_set_velocity(h, v)
    elif call == "step":
        wsb.ws_step(h, 1)
    elif call == "energy":
        assert np.isfinite(wsb.ws_energy(h))
    else:
        wsb.ws_set_storage(h, wsb.WS_STORAGE_FP16)
    for lib in _cudart():       # the caller's own error is the caller's to clear
        lib.cudaGetLastError()
