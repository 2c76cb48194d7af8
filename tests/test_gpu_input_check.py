"""The proper-coloring check of a recoloring input at the row lengths where
its passes change (64/65 entries: lane groups to warps; 4096/4097: warps to
pieces): one same-colored neighbor, wherever it stands in its row, and any
color outside [1, 2^28] make the input improper; the untouched one is taken."""
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

DEGREES = [1, 63, 64, 65, 256, 4095, 4096, 4097, 8192, 8193]


@pytest.fixture(scope="module")
def graph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    g = gg.hubs(DEGREES, 9000, seed=8)
    colors, _ = gc.gc_color(g.offsets.cuda(), g.idx.cuda(), "RXF", 5, 3)
    return g, g.offsets.cuda(), g.idx.cuda(), colors


def _rejected(off, idx, colors):
    for call in (lambda: gc.gc_recolor(off, idx, colors, "RV", 1),
                 lambda: gc.gc_recolor_async(off, idx, colors, "RV", 1),
                 lambda: gc.gc_recolor_batch(off, idx, [dict(n=off.numel() - 1, iterations=1)], colors)):
        with pytest.raises(gc.GCError) as e:
            call()
        assert e.value.name == "GC_ERR_IMPROPER_INPUT"


@pytest.mark.parametrize("hub", range(len(DEGREES)))
@pytest.mark.parametrize("where", ["first", "middle", "last"])
def test_one_conflict_in_a_row(graph, hub, where):
    g, off, idx, colors = graph
    deg = DEGREES[hub]
    at = int(g.offsets[hub]) + {"first": 0, "middle": deg // 2, "last": deg - 1}[where]
    u = int(g.idx[at])
    bad = colors.clone()
    bad[u] = bad[hub]
    _rejected(off, idx, bad)


@pytest.mark.parametrize("color", [0, -3, (1 << 28) + 1])
def test_a_color_out_of_range(graph, color):
    _, off, idx, colors = graph
    bad = colors.clone()
    bad[17] = color
    _rejected(off, idx, bad)


def test_a_proper_input_is_taken(graph):
    _, off, idx, colors = graph
    out, counts, _ = gc.gc_recolor(off, idx, colors, "RV", 2)
    assert counts[0] == int(colors.max()) and counts[2] <= counts[0]
    big = colors.clone()
    big[17] = 1 << 12
    assert gc.gc_recolor(off, idx, big, "RV", 1)[1][0] == 1 << 12
