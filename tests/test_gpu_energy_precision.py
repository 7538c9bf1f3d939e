"""The energy's precision on small and uneven fields (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402

C = [np.longdouble(-205) / 72, np.longdouble(8) / 5, np.longdouble(-1) / 5,
     np.longdouble(8) / 315, np.longdouble(-1) / 560]
H, DT = 10.0, 0.4 * 10.0 / 4500.0


def reference(u, p, v):
    """The energy and the sum of its parts' magnitudes, in the longest float."""
    r = v.astype(np.float64) * (DT / H)
    w = (r * r).astype(np.float32).astype(np.longdouble)
    u, p = (x.astype(np.longdouble) for x in (u, p))
    pad = np.pad(p, 4)
    core = tuple(slice(4, 4 + n) for n in p.shape)
    lap, mag = 3 * C[0] * p, -3 * C[0] * np.abs(p)
    for d in range(3):
        for m in range(1, 5):
            for s in (m, -m):
                sl = list(core)
                sl[d] = slice(4 + s, 4 + s + p.shape[d])
                lap = lap + C[m] * pad[tuple(sl)]
                mag = mag + np.abs(C[m] * pad[tuple(sl)])
    kin = (u - p) ** 2 / (w * H * H)
    return (kin - u * lap / (H * H)).sum(), (kin + np.abs(u) * mag / (H * H)).sum()


def energy(u, p, v):
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    wsb.ws_energy_noalloc(*(torch.from_numpy(x).cuda() for x in (u, p, v)), H, DT, out)
    return float(out[0])


@pytest.mark.parametrize("shape,count", [((1, 1, 1), 300), ((2, 3, 2), 100), ((4, 4, 4), 60),
                                         ((7, 8, 9), 30), ((3, 41, 35), 6)])
@pytest.mark.parametrize("kind", ["alike", "wide", "spike"])
def test_energy_is_as_precise_as_doubles(shape, count, kind):
    """On small grids, where no average hides it, and with values of one size, of
    very different sizes, and single large ones: within the bound of an
    evaluation in doubles. u = 2^-53: a term and its place in the sum take at
    most 8 roundings (a single cell), and with more cells the rows of a thread,
    the block's and the last sum 16 more, each at most u of the parts'
    magnitudes."""
    rng = np.random.default_rng([len(kind), *shape])
    worst = 0.0
    for _ in range(count):
        u = rng.standard_normal(shape)
        p = u + 0.3 * rng.standard_normal(shape)
        if kind == "wide":
            amp = np.exp(8 * rng.standard_normal(shape))
            u, p = u * amp / amp.max(), p * amp / amp.max()
        if kind == "spike":
            amp = np.where(rng.random(shape) < 0.02, 1.0, 2.0 ** -25)
            u, p = u * amp, p * amp
        u, p = u.astype(np.float32), p.astype(np.float32)
        v = rng.uniform(1500.0, 4500.0, shape).astype(np.float32)
        ref, mag = reference(u, p, v)
        worst = max(worst, float(abs(energy(u, p, v) - ref) / mag))
    assert worst <= (8 if shape == (1, 1, 1) else 24) * 2.0 ** -53, worst * 2.0 ** 53
