"""The energy over the ranges and shapes where its summation changes form."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402

C = [np.longdouble(-205) / 72, np.longdouble(8) / 5, np.longdouble(-1) / 5,
     np.longdouble(8) / 315, np.longdouble(-1) / 560]


def energy(u, p, w, h):
    """The definition in the longest float numpy has; w is the stored model."""
    u, p, w = (x.astype(np.longdouble) for x in (u, p, w))
    pad = np.pad(p, 4)
    core = tuple(slice(4, 4 + n) for n in p.shape)
    lap = 3 * C[0] * p
    for d in range(3):
        for m in range(1, 5):
            for s in (m, -m):
                sl = list(core)
                sl[d] = slice(4 + s, 4 + s + p.shape[d])
                lap = lap + C[m] * pad[tuple(sl)]
    return float(((u - p) ** 2 / (w * h * h) - u * lap / (h * h)).sum())


def model(v, dt, h):
    r = v.astype(np.float64) * (dt / h)
    return (r * r).astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 7), (9, 33, 31), (6, 40, 70), (12, 64, 129)])
@pytest.mark.parametrize("scale", ["one", "tiny", "huge", "denormal", "mixed", "quiet", "slow"])
def test_energy_ranges(shape, scale):
    """Amplitudes from denormal to 1e15, blocks of very different size, quiet
    blocks, and models below the two-float form's range; both entry points
    give one value. Bound: every form's terms are within 2^-44 of theirs
    (n-term sums of pairs of floats and of doubles), so 1e-13 of the sum of the
    terms' magnitudes, which is at most a few times the energy here."""
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    u = rng.standard_normal(shape)
    p = u + 0.3 * rng.standard_normal(shape)
    amp = {"tiny": 1e-25, "huge": 1e15, "denormal": 1e-39}.get(scale, 1.0)
    if scale == "mixed":
        amp = 10.0 ** (-30.0 * (np.arange(nz)[:, None, None] % 2))
    if scale == "quiet":
        amp = (np.arange(ny)[None, :, None] < 32).astype(float)
    u, p = (u * amp).astype(np.float32), (p * amp).astype(np.float32)
    h, dt = 10.0, 0.4 * 10.0 / 4500.0
    v = rng.uniform(1500.0, 4500.0, shape).astype(np.float32)
    if scale == "slow":
        v[rng.random(shape) < 0.02] = 1e-7
    hd = wsb.ws_create(nx, ny, nz, h, dt)
    wsb.ws_set_velocity(hd, v)
    wsb.ws_write_field(hd, u, p, 0)
    e = wsb.ws_energy(hd)
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    wsb.ws_energy_noalloc(*(torch.from_numpy(x).cuda() for x in (u, p, v)), h, dt, out)
    assert float(out[0]) == e
    ref = energy(u, p, model(v, dt, h), h)
    assert abs(e - ref) <= 1e-13 * abs(ref)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_energy_of_a_field_that_is_not_finite(bad):
    shape = (5, 40, 40)
    rng = np.random.default_rng(3)
    u, p = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    hd = wsb.ws_create(40, 40, 5, 10.0, 0.4 * 10.0 / 4500.0)
    wsb.ws_set_velocity(hd, np.full(shape, 3000.0, np.float32))
    u[2, 35, 39] = bad
    wsb.ws_write_field(hd, u, p, 0)
    assert not np.isfinite(wsb.ws_energy(hd))
