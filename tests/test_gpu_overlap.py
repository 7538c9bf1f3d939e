"""Steps whose launches overlap, in company (GPU).

A step may start while the one before it still runs; other handles' steps, copies
and cleared fields on the same stream, or a graph that replays the launches, must
not change a bit.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_03775_gb300 as wsb  # noqa: E402
from paper_2204_03775_gb300 import synthetic  # noqa: E402

# (nz, ny, nx), storage: the direct kernel, the streaming one, 16-bit fields
KINDS = [((30, 40, 50), wsb.WS_STORAGE_FP32), ((50, 70, 130), wsb.WS_STORAGE_FP32),
         ((40, 64, 100), wsb.WS_STORAGE_FP16)]


def _handle(kind, stream, sources=True):
    (nz, ny, nx), storage = kind
    h = wsb.ws_create(nx, ny, nz, 10.0, synthetic.cfl_dt(4500.0, 10.0))
    wsb.ws_set_stream(h, stream)
    wsb.ws_set_storage(h, storage)
    wsb.ws_set_velocity(h, synthetic.smooth_random_velocity((nz, ny, nx), nx, 1500.0, 4500.0, spacing=4))
    wsb.ws_set_sponge(h, 4, 0.1)
    if sources:
        wsb.ws_add_source(h, nx // 2, ny // 2, nz // 2, 30.0, 0.0, 1.0)
        wsb.ws_add_source(h, 1, 2, 3, 25.0, 0.01, 2.0)
    return h


def _receivers(kind, seed, n):
    nz, ny, nx = kind[0]
    rng = np.random.default_rng(seed)
    return np.stack([rng.integers(0, m, n) for m in (nx, ny, nz)], 1).astype(np.int32)


def test_handles_that_take_turns_on_one_stream():
    """Three handles step by step on one stream, each with its receivers set anew
    (as many as before) and its field put back from its own arrays now and then,
    without a wait: the bits of each handle alone."""
    stream = torch.cuda.Stream()

    def work(h, kind, turn, kept):
        if turn == 0:
            wsb.ws_set_receivers(h, _receivers(kind, 0, 40), 60)
        if turn in (7, 8, 20):
            wsb.ws_set_receivers(h, _receivers(kind, turn, 40), 60)
        if turn == 12:
            wsb.ws_read_field(h, *kept[:2])
            wsb.ws_write_field(h, None, None, 12)
            wsb.ws_step(h, 1)
            wsb.ws_write_field(h, *kept[:2], 12)
            wsb.ws_set_receivers(h, _receivers(kind, 99, 40), 60)
        wsb.ws_step(h, 1 + turn % 2)
        if turn == 29:
            wsb.ws_read_field(h, *kept[2:4])
            wsb.ws_read_traces(h, kept[4])

    def buffers(kind):
        return [torch.empty(kind[0], device="cuda") for _ in range(4)] + [torch.empty((40, 60), device="cuda")]

    together = [(_handle(k, stream), k, buffers(k)) for k in KINDS]
    for turn in range(30):
        for h, k, kept in together:
            work(h, k, turn, kept)
    torch.cuda.synchronize()
    for h, k, kept in together:
        alone, ref = _handle(k, torch.cuda.Stream()), buffers(k)
        for turn in range(30):
            work(alone, k, turn, ref)
            wsb.ws_synchronize(alone)
        for a, b in zip(kept, ref):
            assert float(b.abs().max()) > 0
            assert torch.equal(a, b)


@pytest.mark.parametrize("kind", KINDS)
def test_steps_in_a_callers_graph(kind):
    """Four steps captured by the caller and replayed are those steps again (no
    sources: their samples belong to the step; four, the cycle of the 16-bit
    state's scales)."""
    stream = torch.cuda.Stream()
    u, p = (torch.from_numpy(np.random.default_rng(s).standard_normal(kind[0]).astype(np.float32)).cuda()
            for s in (1, 2))
    p = u + 0.1 * p
    torch.cuda.synchronize()
    h, ref = (_handle(kind, s, sources=False) for s in (stream, torch.cuda.Stream()))
    for x in (h, ref):
        wsb.ws_write_field(x, u, p, 0)
        wsb.ws_step(x, 4)
        wsb.ws_synchronize(x)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        wsb.ws_step(h, 4)
    with torch.cuda.stream(stream):
        for _ in range(5):
            graph.replay()
    torch.cuda.synchronize()
    wsb.ws_step(ref, 20)
    for a, b in zip(wsb.ws_read_field(h), wsb.ws_read_field(ref)):
        assert np.abs(b).max() > 0
        assert np.array_equal(a, b)
