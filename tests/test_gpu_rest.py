"""Fields from rest, small and large (GPU)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402


@pytest.mark.parametrize("shape", [(24, 500, 300), (64, 800, 800)])
def test_fields_from_rest(shape):
    """Fields below and above the size from which memsets clear them: whatever
    level is missing is zero, the other one what was written."""
    nz, ny, nx = shape
    u, p = (torch.randn(shape, device="cuda") for _ in range(2))
    zero = torch.zeros_like(u)
    out = [torch.empty_like(u) for _ in range(2)]
    torch.cuda.synchronize()
    h = wsb.ws_create(nx, ny, nz, 1.0, 1e-5)
    for levels in ((u, p), (None, None), (u, p), (u, None), (u, p), (None, p)):
        wsb.ws_write_field(h, *levels, 0)
        wsb.ws_read_field(h, *out)
        wsb.ws_synchronize(h)
        for a, b in zip(out, levels):
            assert torch.equal(a, zero if b is None else b)
