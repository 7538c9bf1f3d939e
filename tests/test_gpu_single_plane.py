"""Host copies of grids of one plane (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402


@pytest.mark.parametrize("shape", [(1, 40, 300), (1, 300, 40), (1, 1, 256), (1, 1, 255), (2, 3, 300)])
def test_single_planes_to_the_host(shape):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    u, p = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 1.0, 1e-5)
    wsb.ws_test_fill_padding(h)
    wsb.ws_write_field(h, u, p, 0)
    for a, b in zip(wsb.ws_read_field(h), (u, p)):
        assert np.array_equal(a, b)
    assert wsb.ws_test_check_padding(h) == 0
