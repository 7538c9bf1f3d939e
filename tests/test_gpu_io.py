"""State copies between user arrays and the padded fields (GPU).

Device arrays go through the copy kernels, host arrays through plane copies;
the two must agree byte for byte, whatever the row length (whole vectors, a
ragged tail, single cells), the alignment of the device array, one field or
both, and nothing outside the interior may change.
"""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402
from paper_2204_03775_gb300 import binding  # noqa: E402


def device_copy(a, offset):
    """The array on the GPU, its first element `offset` elements into an allocation."""
    t = torch.empty(a.size + offset, dtype=torch.float32, device="cuda")
    v = t[offset:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 2, 3), (2, 5, 4), (7, 3, 36), (5, 9, 101),
                                   (4, 33, 130), (3, 8, 1028), (6, 400, 64)])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_device_copies_equal_host_copies(shape, offset):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    u, p = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_test_fill_padding(h)
    du, dp = device_copy(u, offset), device_copy(p, offset)
    for first, second in ((u, p), (u, None), (None, p)):
        wsb.ws_write_field(h, None, None, 0)
        wsb.ws_write_field(h, None if first is None else du, None if second is None else dp, 0)
        ref = [np.zeros(shape, np.float32) if a is None else a for a in (first, second)]
        hu, hp = wsb.ws_read_field(h)          # host copies
        assert np.array_equal(hu, ref[0]) and np.array_equal(hp, ref[1])
        ou, op = device_copy(np.full(shape, 7, np.float32), offset), \
            device_copy(np.full(shape, 7, np.float32), offset)
        wsb.ws_read_field(h, ou, op)
        assert np.array_equal(ou.cpu().numpy(), ref[0]) and np.array_equal(op.cpu().numpy(), ref[1])
        ou.fill_(7)
        wsb.ws_read_field(h, None, ou, new=False)
        assert np.array_equal(ou.cpu().numpy(), ref[1])
    # the same array for both levels: the copies run one after the other
    wsb.ws_write_field(h, du, dp, 0)
    wsb.ws_read_field(h, ou, ou)
    assert np.array_equal(ou.cpu().numpy(), p)
    # nothing outside the interior was written
    wsb.ws_test_fill_padding(h)
    wsb.ws_write_field(h, du, dp, 0)
    assert wsb.ws_test_check_padding(h) == 0


def near_ties(values, of):
    """The values whose double result lies closest to the middle of two floats."""
    x = of(values.astype(np.float64))
    f = x.astype(np.float32)
    gap = np.abs(np.abs(x - f.astype(np.float64)) - 0.5 * np.spacing(f).astype(np.float64))
    return values[np.argsort(gap / x)[:8]]


@pytest.mark.parametrize("slowness", [False, True])
@pytest.mark.parametrize("nx,offset", [(64, 0), (64, 1), (67, 0), (5, 0)])
def test_model_is_the_rounded_double(slowness, nx, offset):
    """The stored model is (V dt/h)^2, formed in double and rounded once, also
    where the double lies next to a tie between two floats: read back exactly
    as one step from rest under sources of amplitude 1 with h = 1."""
    ny, nz, dt = 3, 5, 0.4 / 4500.0
    rng = np.random.default_rng(nx + offset)
    many = rng.uniform(1500.0, 4500.0, 1 << 20).astype(np.float32)
    if slowness:
        many = (1.0 / many.astype(np.float64) ** 2).astype(np.float32)
        of = lambda m: (dt * dt) / m                      # noqa: E731
    else:
        of = lambda v: (v * dt) * (v * dt)                # noqa: E731
    vals = np.concatenate([near_ties(many, of), many[:8]])
    model = np.full((nz, ny, nx), vals[0], np.float32)
    cells = [tuple(int(c) for c in np.unravel_index(q, model.shape))
             for q in rng.choice(model.size, 16, replace=False)]
    cells[0] = (nz - 1, ny - 1, nx - 1)
    for c, v in zip(cells, vals):
        model[c] = v
    expected = np.zeros(model.shape, np.float32)
    for c in set(cells):
        expected[c] = np.float32(of(np.float64(model[c])))
    for on_device in (True, False):
        h = wsb.ws_create(nx, ny, nz, 1.0, dt)
        wsb.ws_test_fill_padding(h)
        setter = wsb.ws_set_slowness2 if slowness else wsb.ws_set_velocity
        setter(h, device_copy(model, offset) if on_device else model)
        for k, j, i in set(cells):
            wsb.ws_add_source(h, i, j, k, 10.0, 0.0, 1.0)
        wsb.ws_step(h, 1)
        u, _ = wsb.ws_read_field(h)
        assert np.array_equal(u, expected)
        assert wsb.ws_test_check_padding(h) == 0
        bad = model.copy()
        bad[nz // 2, 0, nx - 1] = np.nan
        with pytest.raises(wsb.WaveStepError):
            setter(h, device_copy(bad, offset) if on_device else bad)


@pytest.mark.parametrize("storage", [wsb.WS_STORAGE_FP16, wsb.WS_STORAGE_BF16])
@pytest.mark.parametrize("nx,offset", [(64, 0), (64, 1), (67, 0), (130, 2), (101, 3)])
def test_16bit_state_of_device_and_host_arrays(storage, nx, offset):
    """The 16-bit state made from device arrays is the one made from host
    arrays, and comes back alike to both; a missing level counts as zero."""
    shape = (5, 17, nx)
    nz, ny, _ = shape
    rng = np.random.default_rng(nx)
    u, p = (rng.standard_normal(shape).astype(np.float32) * 0.3 for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_set_storage(h, storage)
    wsb.ws_test_fill_padding(h)
    du, dp = device_copy(u, offset), device_copy(p, offset)
    zero = np.zeros(shape, np.float32)
    for first, second, hf, hs in ((du, dp, u, p), (du, None, u, zero), (None, dp, zero, p)):
        wsb.ws_write_field(h, hf, hs, 5)
        wsb.ws_test_fill_padding(h)
        ref = wsb.ws_read_field(h)
        assert np.abs(ref[0] - hf).max() < 4e-3
        wsb.ws_write_field(h, first, second, 6)
        got = wsb.ws_read_field(h)
        ou, op = (device_copy(np.full(shape, 7, np.float32), offset) for _ in range(2))
        wsb.ws_read_field(h, ou, op)
        for r, g, o in zip(ref, got, (ou, op)):
            assert np.array_equal(r, g) and np.array_equal(r, o.cpu().numpy())
        wsb.ws_read_field(h, ou, ou)
        assert np.array_equal(ou.cpu().numpy(), ref[1])
        assert wsb.ws_test_check_padding(h) == 0


def test_host_arrays_larger_than_the_staging():
    """Host arrays move through the device staging in groups of planes: a field
    of several groups, the last one short, comes back byte for byte."""
    nz, ny, nx = 19, 1500, 1001       # 6 MB a plane, 10 planes in 64 MiB
    rng = np.random.default_rng(0)
    u, p = (rng.standard_normal((nz, ny, nx)).astype(np.float32) for _ in range(2))
    h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
    wsb.ws_write_field(h, u, p, 0)
    du, dp = device_copy(np.zeros_like(u), 0), device_copy(np.zeros_like(u), 0)
    wsb.ws_read_field(h, du, dp)
    assert np.array_equal(du.cpu().numpy(), u) and np.array_equal(dp.cpu().numpy(), p)
    hu, hp = wsb.ws_read_field(h)
    assert np.array_equal(hu, u) and np.array_equal(hp, p)
    assert wsb.ws_test_check_padding(h) >= 0


def test_receivers_set_again_and_again():
    """Receiver buffers are kept while large enough: fewer, more, none, and the
    same again give the traces of a new handle each time."""
    nx, ny, nz = 70, 30, 20
    v = np.full((nz, ny, nx), 3000.0, np.float32)

    def handle():
        h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
        wsb.ws_set_velocity(h, v)
        wsb.ws_add_source(h, 30, 15, 10, 40.0, 0.0, 1.0)
        return h

    rng = np.random.default_rng(1)
    kept = handle()
    for nrec, nt in ((5, 8), (200, 20), (3, 4), (0, 0), (90, 12), (200, 20)):
        rec = np.stack([rng.integers(0, n, nrec) for n in (nx, ny, nz)], 1).astype(np.int32)
        new = handle()
        for h in (kept, new):
            wsb.ws_write_field(h, None, None, 0)
            wsb.ws_set_receivers(h, rec, nt)
            wsb.ws_step(h, max(nt, 3) - 1)
        a, b = wsb.ws_read_traces(kept), wsb.ws_read_traces(new)
        assert np.array_equal(a, b) and (nrec == 0 or not a[:, -1].any())


@pytest.mark.parametrize("kind", ["bytes", "pinned"])
@pytest.mark.parametrize("storage", [wsb.WS_STORAGE_FP32, wsb.WS_STORAGE_FP16])
def test_arrays_that_no_kernel_may_take(kind, storage):
    """Arrays said to be on the device that are not float-aligned, or lie in
    host memory, go through the copies that take any address: right or refused."""
    lib = binding.load_library()
    shape = (5, 17, 67)
    nz, ny, nx = shape
    rng = np.random.default_rng(3)
    u = rng.integers(-64, 64, shape).astype(np.float32)
    v = np.full(shape, 3000.0, np.float32)

    def handle():
        h = wsb.ws_create(nx, ny, nz, 10.0, 1e-3)
        wsb.ws_set_storage(h, storage)
        return h

    if kind == "bytes":
        raw = [torch.zeros(u.nbytes + 2, dtype=torch.uint8, device="cuda") for _ in range(3)]
        views = [r[2:] for r in raw]
    else:
        views = [torch.zeros(u.nbytes, dtype=torch.uint8).pin_memory() for _ in range(3)]
    for t, a in zip(views, (u, v)):
        t.copy_(torch.from_numpy(a.reshape(-1).view(np.uint8).copy()))
    torch.cuda.synchronize()
    pu, pv, po = (ctypes.c_void_p(t.data_ptr()) for t in views)
    h, ref = handle(), handle()
    wsb.ws_write_field(ref, u, None, 0)
    wsb.ws_set_velocity(ref, v)
    ok = [lib.ws_write_field(h.ptr, pu, None, 0, 1), lib.ws_set_velocity(h.ptr, pv, 1),
          lib.ws_read_field(ref.ptr, po, None, 1)]
    wsb.ws_synchronize(h)
    wsb.ws_synchronize(ref)
    if kind == "bytes":
        assert ok == [0, 0, 0]
    if ok[0] == 0 and ok[1] == 0:
        for g in (h, ref):
            wsb.ws_step(g, 2)
        assert all(np.array_equal(a, b) for a, b in zip(wsb.ws_read_field(h), wsb.ws_read_field(ref)))
    if ok[2] == 0:
        assert np.array_equal(views[2].cpu().numpy().view(np.float32).reshape(shape), u)
