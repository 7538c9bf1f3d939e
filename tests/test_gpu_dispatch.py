"""Kernel and tiling choice (GPU): whatever kernel, tile and z block a step
takes, the fields and the traces are the same bits."""

import numpy as np
import pytest

import paper_2204_03775_gb300 as wsb
from paper_2204_03775_gb300 import synthetic

pytestmark = pytest.mark.gpu

NT = 14


def _run(shape, kernel, tile=(0, 0), zblock=0):
    """Fields and traces after NT steps of a tapered model with sources and
    receivers on faces, edges, tile borders and in one column."""
    nz, ny, nx = shape
    vel = synthetic.smooth_random_velocity(shape, 11, 1500.0, 4500.0, spacing=4)
    h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
    wsb.ws_set_kernel(h, kernel, *tile, zblock)
    wsb.ws_set_velocity(h, vel)
    wsb.ws_set_sponge(h, 3, 0.2)
    cells = [(0, 0, 0), (nx - 1, ny - 1, nz - 1), (nx // 2, ny // 2, nz // 2),
             (min(63, nx - 1), min(15, ny - 1), 0), (min(64, nx - 1), min(16, ny - 1), nz - 1),
             (nx // 2, min(7, ny - 1), nz // 3), (nx // 2, min(8, ny - 1), nz // 3)]
    for n, c in enumerate(cells):
        wsb.ws_add_source(h, *c, 20.0, 0.01 + 0.001 * n, 1.0 + n)
    rec = cells + cells[:2] + [(nx // 2, ny // 2, k) for k in range(nz)] \
        + [(i, ny // 2, nz // 2) for i in range(0, nx, 3)]
    wsb.ws_set_receivers(h, np.array(rec, np.int32), NT)
    wsb.ws_step(h, 5)
    wsb.ws_step(h, NT - 5)
    wsb.ws_synchronize(h)
    u, p = wsb.ws_read_field(h)
    return u, p, wsb.ws_read_traces(h)


@pytest.mark.parametrize("tile", [(64, 16), (64, 8), (64, 32), (32, 16), (32, 8)])
@pytest.mark.parametrize("shape", [(9, 32, 64), (10, 33, 65), (13, 47, 131), (5, 34, 98)])
def test_every_tile_gives_the_direct_kernels_bits(tile, shape):
    ref = _run(shape, wsb.WS_KERNEL_DIRECT)
    assert np.abs(ref[2]).max() > 0
    for zblock in (0, 1, 2, 3, 4, 7, shape[0]):
        for r, x in zip(ref, _run(shape, wsb.WS_KERNEL_STREAM, tile, zblock)):
            assert np.array_equal(r, x)


@pytest.mark.parametrize("shape", [(15, 99, 101), (15, 100, 101), (20, 100, 101), (40, 40, 48), (6, 12, 80),
                                   (7, 40, 33), (3, 5, 300)])
def test_default_choice_gives_the_direct_kernels_bits(shape):
    """Grids on both sides of the direct kernel's limit, low and narrow ones."""
    ref = _run(shape, wsb.WS_KERNEL_DIRECT)
    for r, x in zip(ref, _run(shape, wsb.WS_KERNEL_AUTO)):
        assert np.array_equal(r, x)
    nz, ny, nx = shape
    if nx >= 64 and ny >= 8:      # STREAM without a tile needs 64 x 8, as ever
        for r, x in zip(ref, _run(shape, wsb.WS_KERNEL_STREAM)):
            assert np.array_equal(r, x)
    else:
        h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
        with pytest.raises(wsb.WaveStepError):
            wsb.ws_set_kernel(h, wsb.WS_KERNEL_STREAM)


@pytest.mark.parametrize("nt", [1, 2, 3, 4, 5, 7, 8, 10])
@pytest.mark.parametrize("shape", [(12, 20, 40), (20, 100, 130)])
def test_forward_run_for_every_segment_length(nt, shape):
    """ws_forward keeps its checkpoints where its steps wrote them: whatever the
    length of the last segment (one step, a whole one), state and traces are
    those of ws_step, and a gradient that reuses the run twice is the one that
    makes its own. Direct and streaming kernel; receivers share cells, one lies on
    the source (else one step has no gradient)."""
    nz, ny, nx = shape
    vel = synthetic.smooth_random_velocity(shape, 5, 1500.0, 4500.0, spacing=4)
    dt = synthetic.cfl_dt(4500.0, 10.0)
    rec = np.array([[5, 5, 3], [3, 4, 2], [3, 4, 2], [nx - 1, ny - 1, nz - 1], [0, 0, 0]]
                   + [[i, 9, 2] for i in range(0, nx, 2)], np.int32)
    r = np.random.default_rng(nt).standard_normal((len(rec), nt)).astype(np.float32)

    def handle():
        h = wsb.ws_create(nx, ny, nz, 10.0, dt)
        wsb.ws_set_velocity(h, vel)
        wsb.ws_set_sponge(h, 3, 0.1)
        wsb.ws_add_source(h, 5, 5, 3, 30.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, rec, nt)
        return h

    a, b, c = handle(), handle(), handle()
    wsb.ws_step(a, nt)
    wsb.ws_forward(b)
    for x, y in zip(wsb.ws_read_field(a), wsb.ws_read_field(b)):
        assert np.array_equal(x, y)
    assert np.array_equal(wsb.ws_read_traces(a), wsb.ws_read_traces(b))
    own, _ = wsb.ws_adjoint_gradient(c, r, wsb.WS_ADJ_RESIDUAL)
    assert np.abs(own).max() > 0
    for _ in range(2):
        g, _ = wsb.ws_adjoint_gradient(b, r, wsb.WS_ADJ_RESIDUAL)
        # receivers that share a cell may be added in another order
        assert np.abs(g - own).max() <= 1e-6 * np.abs(own).max()


@pytest.mark.parametrize("tile", [(64, 16), (32, 16), (64, 8), (32, 8)])
@pytest.mark.parametrize("shared", [0, 40])
def test_injection_of_dense_receivers(tile, shared):
    """The adjoint step's injection with a receiver on every cell of two planes,
    in no order (8 a thread, 256 a warp): the direct kernel's bits. With 40 more
    on one cell, added in another order, to the rounding of such a sum of
    residuals of one sign (40 half ulps, four times that for the gradient)."""
    shape = nz, ny, nx = 9, 20, 70
    vel = synthetic.smooth_random_velocity(shape, 5, 1500.0, 4500.0, spacing=4)
    rng = np.random.default_rng(shared)
    rec = np.array([[i, j, k] for k in (2, 5) for j in range(ny) for i in range(nx)], np.int32)
    rec = np.concatenate([rec[rng.permutation(len(rec))], np.repeat([[66, 17, 5]], shared, 0)])
    rec = rec.astype(np.int32)
    nt = 5
    r = rng.uniform(0.5, 1.0, (len(rec), nt)).astype(np.float32)
    grads = []
    for kernel, size in ((wsb.WS_KERNEL_DIRECT, (0, 0)), (wsb.WS_KERNEL_STREAM, tile)):
        h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
        wsb.ws_set_kernel(h, kernel, *size, 0)
        wsb.ws_set_velocity(h, vel)
        wsb.ws_set_sponge(h, 3, 0.1)
        wsb.ws_add_source(h, 30, 5, 3, 30.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, rec, nt)
        grads.append(wsb.ws_adjoint_gradient(h, r, wsb.WS_ADJ_RESIDUAL)[0])
    assert np.abs(grads[0]).max() > 0
    if shared:
        assert np.abs(grads[0] - grads[1]).max() <= 4 * 40 * 2.0 ** -24 * np.abs(grads[0]).max()
    else:
        assert np.array_equal(*grads)
