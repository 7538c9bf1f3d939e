"""Device memory that a handle keeps (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402


def test_large_receiver_buffers_are_given_back():
    """Buffers are kept for receivers set again, not a gigabyte of traces under a
    few small ones."""
    nz, ny, nx = 20, 40, 80
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_set_velocity(h, np.full((nz, ny, nx), 3000.0, np.float32))
    few = np.zeros((4, 3), np.int32)
    wsb.ws_set_receivers(h, few, 16)
    wsb.ws_step(h, 1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    wsb.ws_set_receivers(h, np.zeros((256, 3), np.int32), 1 << 20)     # 1 GiB
    wsb.ws_step(h, 1)
    wsb.ws_synchronize(h)
    assert before - torch.cuda.mem_get_info()[0] > 1000 << 20
    wsb.ws_set_receivers(h, few, 16)
    wsb.ws_step(h, 1)
    wsb.ws_synchronize(h)
    assert before - torch.cuda.mem_get_info()[0] < 64 << 20


def test_staging_is_given_back_when_memory_runs_out():
    """The device buffer that host arrays move through is the first to go when an
    allocation of its handle fails; the next host array makes it again."""
    nz, ny, nx = 64, 512, 512       # a field of 64 MiB
    u = np.random.default_rng(0).standard_normal((nz, ny, nx)).astype(np.float32)
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]
    wsb.ws_write_field(h, u, None, 0)
    free.append(torch.cuda.mem_get_info()[0])
    with pytest.raises(wsb.WaveStepError) as e:              # 550 GB of traces
        wsb.ws_set_receivers(h, np.zeros((64, 3), np.int32), 2 ** 31 - 1)
    assert e.value.code == wsb.WS_ERR_OOM
    free.append(torch.cuda.mem_get_info()[0])
    assert free[0] - free[1] >= 64 << 20 and free[2] - free[1] >= 64 << 20
    assert np.array_equal(wsb.ws_read_field(h)[0], u)
