"""Adjoint steps with many receivers on one cell (GPU)."""

import time

import numpy as np
import pytest

import paper_2204_03775_gb300 as wsb
from paper_2204_03775_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,n", [(1, 700), (2, 333), (9, 320), (40, 700)])
def test_shared_cells_are_summed(cells, n):
    """The streaming kernel's gradient with n receivers on few cells of two
    neighbouring planes, in any order, is the direct kernel's to the rounding of
    two sums of at most n residuals of one sign (n half ulps each)."""
    shape = nz, ny, nx = 9, 20, 70
    rng = np.random.default_rng(cells)
    places = np.stack([rng.integers(60, 70, cells), rng.integers(12, 20, cells),
                       rng.integers(4, 6, cells)], 1)
    rec = places[rng.integers(0, cells, n)].astype(np.int32)
    nt = 5
    r = rng.uniform(0.5, 1.0, (n, nt)).astype(np.float32)
    grads = []
    for kernel in (wsb.WS_KERNEL_DIRECT, wsb.WS_KERNEL_STREAM):
        h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
        wsb.ws_set_kernel(h, kernel)
        wsb.ws_set_velocity(h, synthetic.smooth_random_velocity(shape, 5, 1500.0, 4500.0, spacing=4))
        wsb.ws_set_sponge(h, 3, 0.1)
        wsb.ws_add_source(h, 62, 14, 5, 30.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, rec, nt)
        grads.append(wsb.ws_adjoint_gradient(h, r, wsb.WS_ADJ_RESIDUAL)[0])
    scale = np.abs(grads[0]).max()
    assert scale > 0 and np.abs(grads[0] - grads[1]).max() <= 2 * n * 2.0 ** -24 * scale


def test_many_receivers_on_one_cell_are_quick():
    """3000 receivers on one cell of 64^3: a gradient within 10 times its time with
    16 (6; one after the other they took 40 times)."""
    torch = pytest.importorskip("torch")
    n, nt = 64, 25

    def best_ms(rec):
        h = wsb.ws_create(n, n, n, 10.0, 1e-3)
        wsb.ws_set_velocity(h, np.full((n, n, n), 2000.0, np.float32))
        wsb.ws_add_source(h, 32, 32, 32, 10.0, 0.0, 1.0)
        wsb.ws_set_receivers(h, rec, nt)
        d = torch.zeros((len(rec), nt), device="cuda")
        g = torch.empty((n, n, n), device="cuda")
        best = np.inf
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            wsb.ws_adjoint_gradient(h, d, wsb.WS_ADJ_RESIDUAL, g)
            best = min(best, time.perf_counter() - t0)
        return best

    few = best_ms(np.array([[16 * i + 8, 16 * j + 8, 3] for i in range(4) for j in range(4)], np.int32))
    assert best_ms(np.full((3000, 3), 32, np.int32)) < 10 * few
