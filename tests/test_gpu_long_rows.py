"""State and model I/O on grids of few long rows (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402


def _ms(stream, fn, n=5):
    fn()
    best = np.inf
    for _ in range(3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(stream)
        for _ in range(n):
            fn()
        b.record(stream)
        b.synchronize()
        best = min(best, a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("storage", [wsb.WS_STORAGE_FP32, wsb.WS_STORAGE_FP16])
@pytest.mark.parametrize("shape", [(1, 17, 1023), (1, 17, 1024), (2, 16, 2049), (1, 16, 4103), (1, 19, 65000)])
def test_few_long_rows(shape, storage):
    """64 to 256 threads a row: device arrays in and out, aligned or not, are the
    host's, the model is the rounded double at both ends and in the middle of a
    row, and its check sees the last cell."""
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    u, p = (rng.integers(-64, 64, shape).astype(np.float32) / 64 for _ in range(2))
    dt = 0.4 / 4500.0
    v = rng.uniform(1500.0, 4500.0, shape).astype(np.float32)
    h = wsb.ws_create(nx, ny, nz, 1.0, dt)
    wsb.ws_set_storage(h, storage)
    for offset in (0, 1):
        raw = [torch.zeros(u.size + 4, device="cuda") for _ in range(4)]
        du, dp, ou, op = (r[offset:offset + u.size].view(shape) for r in raw)
        du.copy_(torch.from_numpy(u))
        dp.copy_(torch.from_numpy(p))
        torch.cuda.synchronize()
        wsb.ws_write_field(h, du, dp, 0)
        wsb.ws_read_field(h, ou, op)
        hu, hp = wsb.ws_read_field(h)
        assert np.array_equal(ou.cpu().numpy(), hu) and np.array_equal(op.cpu().numpy(), hp)
        tol = 0.0 if storage == wsb.WS_STORAGE_FP32 else 2.0 ** -9
        assert np.abs(hu - u).max() <= tol and np.abs(hp - p).max() <= 4 * tol
    if storage == wsb.WS_STORAGE_FP32:
        cells = [(0, 0), (0, nx - 1), (ny - 1, 0), (ny - 1, nx - 1), (3, nx // 2), (5, 511), (6, 512)]
        for arr in (v, torch.from_numpy(v).cuda()):
            wsb.ws_set_velocity(h, arr)
            wsb.ws_write_field(h, None, None, 0)
            wsb.ws_clear_sources(h)
            expected = np.zeros(shape, np.float32)
            for j, i in cells:
                wsb.ws_add_source(h, i, j, nz - 1, 10.0, 0.0, 1.0)
                expected[nz - 1, j, i] = np.float32((np.float64(v[nz - 1, j, i]) * dt) ** 2)
            wsb.ws_step(h, 1)
            assert np.array_equal(wsb.ws_read_field(h)[0], expected)
        bad = torch.from_numpy(v).cuda()
        bad[-1, -1, -1] = np.nan
        with pytest.raises(wsb.WaveStepError):
            wsb.ws_set_velocity(h, bad)


def test_few_long_rows_are_as_fast_as_2d_copies():
    """27 rows of 65000 cells, both levels: in and out within 45 us each (18 and 20;
    2D copies 59 and 38; with 32 threads a row 91 and 95)."""
    shape = nz, ny, nx = 3, 9, 65000
    stream = torch.cuda.Stream()
    h = wsb.ws_create(nx, ny, nz, 1.0, 1e-5)
    wsb.ws_set_stream(h, stream)
    u, p = (torch.randn(shape, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    assert _ms(stream, lambda: wsb.ws_write_field(h, u, p, 0)) < 0.045
    assert _ms(stream, lambda: wsb.ws_read_field(h, u, p)) < 0.045
