"""The energy's signal of a bad model (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402

H, DT = 10.0, 0.4 * 10.0 / 4500.0


@pytest.mark.parametrize("bad", [0.0, np.nan])
@pytest.mark.parametrize("where", [0, 1])
def test_a_bad_model_under_a_quiet_field_shows(bad, where):
    """A velocity that is zero or not a number makes the energy not a number,
    also where both levels are zero (0 / 0), all of them or in one cell's block."""
    shape = (5, 70, 40)
    u = torch.zeros(shape, device="cuda")
    p = torch.zeros(shape, device="cuda")
    if where:
        u[0, 0, 0] = 1.0
    v = torch.full(shape, 3000.0, device="cuda")
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    wsb.ws_energy_noalloc(u, p, v, H, DT, out)
    assert np.isfinite(float(out[0])) and (float(out[0]) > 0) == bool(where)
    v[3, 66, 39] = bad
    wsb.ws_energy_noalloc(u, p, v, H, DT, out)
    assert np.isnan(float(out[0]))
    v[3, 66, 39] = np.inf                    # 0 / inf: nothing
    wsb.ws_energy_noalloc(u, p, v, H, DT, out)
    assert np.isfinite(float(out[0]))
