"""Malformed ids in graphs that fill the GPU: the rounds kernel's blocks meet
at grid barriers, and all of them have to get there whichever block finds a
bad id first.  A call reports GC_ERR_BAD_GRAPH in the time of a coloring (a
barrier that a block never reached gives up after 2^24 polls, some seconds)."""
import time

import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

LIMIT_S = 0.5  # a good coloring of these graphs takes a few milliseconds


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    yield
    gc.gc_set_tuning()


def _with_bad_entries(g, rows, bad):
    """The graph with one more entry, bad[i], at the end of row rows[i] (the other entries stay symmetric)."""
    dev = g.offsets.device
    more = torch.zeros(g.n, dtype=torch.int64, device=dev)
    more[rows] = 1
    off = torch.zeros_like(g.offsets)
    off[1:] = g.offsets[1:] + more.cumsum(0)
    deg = g.offsets[1:] - g.offsets[:-1]
    row = torch.repeat_interleave(torch.arange(g.n, device=dev), deg)
    idx = torch.empty(g.nnz + rows.numel(), dtype=torch.int32, device=dev)
    idx[torch.arange(g.nnz, device=dev) + (off[:-1] - g.offsets[:-1])[row]] = g.idx
    idx[off[1:][rows] - 1] = bad
    return off, idx


def _damaged(g, where):
    dev = g.offsets.device
    rows = {"first": [0], "last": [g.n - 1], "self-loop": [2]}.get(where, list(range(5, g.n, 1001)))
    rows = torch.tensor(rows, device=dev)
    bad = rows.to(torch.int32) if where == "self-loop" else torch.full_like(rows, g.n, dtype=torch.int32)
    if where == "last":
        bad[:] = -1
    return _with_bad_entries(g, rows, bad)


@pytest.mark.parametrize("knobs", [{}, dict(spec_graph=0)])
@pytest.mark.parametrize("where", ["first", "last", "self-loop", "spread"])
@pytest.mark.parametrize("hubs", [[], [70000, 3000, 300]])
def test_every_block_reaches_the_barriers(hubs, where, knobs):
    g = gg.hubs(hubs, 400_000 - len(hubs), seed=7, device="cuda")
    off, idx = _damaged(g, where)
    want, _ = gc.gc_color(g.offsets, g.idx, "FF", 1, 5)
    gc.gc_set_tuning(**knobs)
    for strategy, X in (("FF", 1), ("RXF", 3)) * 4:
        torch.cuda.synchronize()
        t = time.perf_counter()
        with pytest.raises(gc.GCError) as e:
            gc.gc_color(off, idx, strategy, X, 5)
        assert e.value.name == "GC_ERR_BAD_GRAPH"
        assert time.perf_counter() - t < LIMIT_S
    assert torch.equal(gc.gc_color(g.offsets, g.idx, "FF", 1, 5)[0], want)
