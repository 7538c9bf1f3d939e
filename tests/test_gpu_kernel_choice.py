"""Which kernels a handle accepts (GPU)."""

import numpy as np
import pytest

import paper_2204_03775_gb300 as wsb
from paper_2204_03775_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(20, 40, 40), (220, 40, 40), (30, 9, 33), (700, 9, 60)])
def test_stream_kernel_is_accepted_after_automatic_steps(shape):
    """On a grid narrower than 64 x 8 (but not than 32 x 8) the streaming kernel
    without a tile is refused on a new handle, and accepted once AUTO has
    stepped it: with the tile that AUTO takes."""
    nz, ny, nx = shape
    vel = synthetic.smooth_random_velocity(shape, 11, 1500.0, 4500.0, spacing=4)

    def run(stream):
        h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
        wsb.ws_set_velocity(h, vel)
        wsb.ws_add_source(h, nx // 2, ny // 2, nz // 2, 30.0, 0.0, 1.0)
        if stream:
            with pytest.raises(wsb.WaveStepError):
                wsb.ws_set_kernel(h, wsb.WS_KERNEL_STREAM)
        wsb.ws_step(h, 3)
        if stream:
            wsb.ws_set_kernel(h, wsb.WS_KERNEL_STREAM)
        wsb.ws_step(h, 9)
        return wsb.ws_read_field(h)

    for a, b in zip(run(True), run(False)):
        assert np.abs(b).max() > 0
        assert np.array_equal(a, b)
