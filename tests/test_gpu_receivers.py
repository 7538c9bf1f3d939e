"""Receiver tables that are rebuilt while the stream is busy (GPU)."""

import numpy as np
import pytest

import paper_2204_03775_gb300 as wsb
from paper_2204_03775_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [wsb.WS_KERNEL_STREAM, wsb.WS_KERNEL_DIRECT])
def test_table_rebuilt_behind_a_busy_stream(kernel):
    """A table of 1 MB, set again while some hundred steps are queued: its upload
    may run long after the call that issued it, so the host memory it comes from
    has to live on, whatever the host allocates and writes meanwhile. The traces
    are those of a handle that waits after every call."""
    nz, ny, nx = 96, 256, 256
    nt = 150
    vel = synthetic.smooth_random_velocity((nz, ny, nx), 3, 1500.0, 4500.0, spacing=8)
    cells = [np.array([[i, j, k] for j in range(ny) for i in range(nx)], np.int32) for k in (9, 30, 40)]
    rng = np.random.default_rng(5)
    sets = [c[rng.permutation(len(c))] for c in cells]

    def run(wait):
        h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
        wsb.ws_set_velocity(h, vel)
        wsb.ws_set_kernel(h, kernel)
        wsb.ws_add_source(h, nx // 2, ny // 2, 20, 30.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, sets[0], nt)      # the buffers are made here
        wsb.ws_step(h, 1)
        wsb.ws_synchronize(h)
        for rec in sets[1:]:
            wsb.ws_step(h, nt - 1)
            if wait:
                wsb.ws_synchronize(h)
            wsb.ws_set_receivers(h, rec, nt)
            wsb.ws_step(h, 1)
            if wait:
                wsb.ws_synchronize(h)
            else:                                 # the host reuses its memory
                junk = [np.full(rec.size, -1 - q, np.int32) for q in range(16)]
                del junk
        wsb.ws_step(h, 1)
        return wsb.ws_read_traces(h)[:, :2], wsb.ws_read_field(h)[0]

    for a, b in zip(run(False), run(True)):
        assert np.abs(b).max() > 0
        assert np.array_equal(a, b)


def test_dense_receivers_on_a_narrow_grid():
    """Grids narrower than a streaming tile take the direct kernel whatever their
    size: a receiver on every cell of a vertical plane, some cells shared, is
    sampled right, and costs a step a few times its own time at most (the scan
    of a whole column's receivers for each plane took 19 times)."""
    torch = pytest.importorskip("torch")
    nz, ny, nx = 6000, 120, 20
    nt = 72
    vel = synthetic.smooth_random_velocity((nz, ny, nx), 3, 1500.0, 4500.0, spacing=8)
    rec = np.array([[7, j, k] for k in range(nz) for j in range(ny)]
                   + [[7, 60, 750]] * 700 + [[19, 119, nz - 1], [0, 0, 0]], np.int32)
    rec = rec[np.random.default_rng(2).permutation(len(rec))]
    h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
    wsb.ws_set_velocity(h, vel)
    wsb.ws_add_source(h, 8, 60, 750, 30.0, 0.0, 1.0)
    stream = torch.cuda.Stream()
    wsb.ws_set_stream(h, stream)

    def step_ms():
        wsb.ws_step(h, 4)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(stream)
        wsb.ws_step(h, 16)
        b.record(stream)
        b.synchronize()
        return a.elapsed_time(b) / 16

    bare = min(step_ms() for _ in range(3))
    wsb.ws_write_field(h, None, None, 0)
    wsb.ws_set_receivers(h, rec, nt)
    for t in range(4):
        wsb.ws_step(h, 1)
        u, _ = wsb.ws_read_field(h)
        assert np.array_equal(wsb.ws_read_traces(h)[:, t], u[rec[:, 2], rec[:, 1], rec[:, 0]])
    assert np.abs(u).max() > 0
    assert step_ms() < 8 * bare


@pytest.mark.parametrize("sizes", [[60] * 21, [60, 6000, 60, 60, 6000, 6000, 60, 60, 60, 60, 60, 60, 6000, 60]])
def test_many_tables_behind_a_busy_stream(sizes):
    """More tables than the handle keeps host buffers for, small ones and some of
    more than 64 KB, while steps are queued: each step samples its own cells."""
    torch = pytest.importorskip("torch")
    shape = nz, ny, nx = 128, 256, 256
    rng = np.random.default_rng(1)
    vel = synthetic.smooth_random_velocity(shape, 3, 1500.0, 4500.0, spacing=8)
    recs = [np.stack([rng.integers(0, n, m) for n in (nx, ny, nz)], 1).astype(np.int32) for m in sizes]

    def run(wait):
        h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
        wsb.ws_set_velocity(h, vel)
        for k in (20, 60, 100):
            wsb.ws_add_source(h, nx // 2, ny // 2, k, 30.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, recs[1], 30)      # the largest buffers
        wsb.ws_step(h, 30)
        wsb.ws_synchronize(h)
        out = []
        for rec in recs:
            wsb.ws_set_receivers(h, rec, 30)
            wsb.ws_step(h, 30)
            out.append(torch.empty((len(rec), 30), device="cuda"))
            wsb.ws_read_traces(h, out[-1])
            if wait:
                wsb.ws_synchronize(h)
        wsb.ws_synchronize(h)
        return [t.cpu().numpy() for t in out]

    for a, b in zip(run(False), run(True)):
        assert np.abs(b).max() > 0
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [3000, 257, 256, 200])
def test_receivers_crowded_in_few_columns(n):
    """Ranges by tile only (far more blocks than receivers), one of them longer
    than a block, at its limit, or short: every plane finds its own entries."""
    nz, ny, nx = 6000, 64, 20
    vel = synthetic.smooth_random_velocity((nz, ny, nx), 3, 1500.0, 4500.0, spacing=8)
    rng = np.random.default_rng(n)
    rec = np.stack([rng.integers(5, 9, n), rng.integers(16, 20, n), rng.integers(2900, 3100, n)], 1)
    rec = np.concatenate([rec, [[0, 0, 0], [19, 63, 5999], [6, 17, 0], [6, 17, 5999]]]).astype(np.int32)
    h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
    wsb.ws_set_velocity(h, vel)
    rng = np.random.default_rng(0)
    u = rng.standard_normal((nz, ny, nx)).astype(np.float32)
    wsb.ws_write_field(h, u, u, 0)
    wsb.ws_set_receivers(h, rec, 3)
    for t in range(3):
        wsb.ws_step(h, 1)
        u, _ = wsb.ws_read_field(h)
        assert np.array_equal(wsb.ws_read_traces(h)[:, t], u[rec[:, 2], rec[:, 1], rec[:, 0]])


def test_setting_many_receivers_is_quick():
    """40000 receivers set anew and one step, on a grid that takes the direct
    kernel (whose table once was the list of cells) and on one of the streaming
    kernel: within 1 ms (0.25 and 0.4; sorting them by comparisons took 2.5)."""
    import time
    for shape in ((300, 30, 24), (100, 100, 100)):
        nz, ny, nx = shape
        rng = np.random.default_rng(0)
        rec = rng.integers(0, [nx, ny, nz], (40000, 3)).astype(np.int32)
        h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
        wsb.ws_set_velocity(h, np.full(shape, 2000.0, np.float32))
        best = np.inf
        for _ in range(6):
            wsb.ws_synchronize(h)
            t0 = time.perf_counter()
            wsb.ws_set_receivers(h, rec, 4)
            wsb.ws_step(h, 1)
            wsb.ws_synchronize(h)
            best = min(best, time.perf_counter() - t0)
        assert best < 1e-3, best


def test_dense_receivers_add_little_to_a_step():
    """A receiver on each cell of a vertical plane of a narrow grid: a step within
    1.5 times its time without (1.24; searching each tile's range 1.8)."""
    torch = pytest.importorskip("torch")
    nz, ny, nx = 6000, 120, 20
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_set_velocity(h, np.full((nz, ny, nx), 2000.0, np.float32))
    stream = torch.cuda.Stream()
    wsb.ws_set_stream(h, stream)

    def step_ms():
        wsb.ws_step(h, 4)
        best = np.inf
        for _ in range(3):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(stream)
            wsb.ws_step(h, 12)
            b.record(stream)
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 12)
        return best

    bare = step_ms()
    rec = np.array([[7, j, k] for k in range(nz) for j in range(ny)], np.int32)
    wsb.ws_set_receivers(h, rec, 40)
    assert step_ms() < 1.5 * bare
