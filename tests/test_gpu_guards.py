"""Copies write the cells they are to write and no others (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402

GUARD = 64


def guarded(shape, offset):
    """A device array with cells of a known value on both sides, its start `offset`
    elements behind a 16-byte boundary."""
    n = int(np.prod(shape))
    whole = torch.full((n + 2 * GUARD + offset,), 7.25, device="cuda")
    return whole, whole[GUARD + offset:GUARD + offset + n].view(shape)


def intact(whole, view):
    n, at = view.numel(), view.storage_offset()
    return bool((whole[:at] == 7.25).all()) and bool((whole[at + n:] == 7.25).all())


@pytest.mark.parametrize("storage", [wsb.WS_STORAGE_FP32, wsb.WS_STORAGE_FP16, wsb.WS_STORAGE_BF16])
@pytest.mark.parametrize("nx", [64, 65, 66, 67, 131])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_nothing_around_the_callers_arrays_is_written(storage, nx, offset):
    shape = nz, ny, _ = 3, 17, nx
    rng = np.random.default_rng(nx)
    u, p = (rng.integers(-64, 64, shape).astype(np.float32) / 64 for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_set_storage(h, storage)
    wsb.ws_set_velocity(h, np.full(shape, 3000.0, np.float32))
    wsb.ws_set_receivers(h, np.array([[nx - 1, ny - 1, nz - 1], [0, 0, 0], [5, 5, 1]], np.int32), 5)
    wsb.ws_write_field(h, u, p, 0)
    (wu, vu), (wp, vp), (wt, vt) = guarded(shape, offset), guarded(shape, 3 - offset), guarded((3, 5), offset)
    wsb.ws_read_field(h, vu, vp)
    wsb.ws_read_traces(h, vt)
    wsb.ws_synchronize(h)
    ref = wsb.ws_read_field(h)
    assert np.abs(ref[0] - u).max() <= 2.0 ** -8 and np.abs(ref[1] - p).max() <= 2.0 ** -6
    assert np.array_equal(vu.cpu().numpy(), ref[0]) and np.array_equal(vp.cpu().numpy(), ref[1])
    assert intact(wu, vu) and intact(wp, vp) and intact(wt, vt)
    wu.fill_(7.25)
    wsb.ws_read_field(h, vu, None)
    wsb.ws_synchronize(h)
    assert intact(wu, vu) and np.array_equal(vu.cpu().numpy(), ref[0])


def test_staged_planes_stay_in_the_interior():
    """Host arrays of several groups of planes, with canaries around every row: a
    state in and out, a model, and nothing else touched."""
    nz, ny, nx = 19, 1500, 1001       # 6 MB a plane, 10 planes in 64 MiB
    rng = np.random.default_rng(0)
    u, p = (rng.standard_normal((nz, ny, nx)).astype(np.float32) for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_test_fill_padding(h)
    wsb.ws_write_field(h, u, p, 0)
    wsb.ws_set_velocity(h, np.full((nz, ny, nx), 3000.0, np.float32))
    assert wsb.ws_test_check_padding(h) == 0
    for a, b in zip(wsb.ws_read_field(h), (u, p)):
        assert np.array_equal(a, b)
    assert wsb.ws_test_check_padding(h) == 0
