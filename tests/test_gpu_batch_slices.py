"""The per-vertex passes of a batch, which take slices of 2048 vertices: class
tables at and beyond what a block counts in shared memory (512 classes),
hundreds of graphs in a slice, empty graphs at its ends, graphs over several
slices; each equals the oracle's coloring and recoloring of it alone."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

BATCHES = {
    "512 classes": lambda: [gg.complete(511)],
    "513 classes": lambda: [gg.complete(512)],
    "two tables": lambda: [gg.complete(200), gg.empty(1000), gg.complete(310), gg.erdos_renyi(3000, 9.0, 1)],
    "many small": lambda: [gg.path(1 + i % 4) for i in range(1500)],
    "empty ends": lambda: [gg.empty(0), gg.grid_2d(64, 32), gg.empty(0), gg.empty(0), gg.cycle(2048), gg.empty(0)],
    "long": lambda: [gg.hubs([600, 900], 5001, seed=2), gg.erdos_renyi(2047, 5.0, 4), gg.empty(4099)],
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_slices(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    graphs = BATCHES[name]()
    desc = [dict(n=g.n, seed=11 + i, X=1 + 3 * (i % 2), perm=["ND", "RAND", "RV"][i % 3], iterations=i % 4 + 1,
                 perm_seed=i) for i, g in enumerate(graphs)]
    u = gg.batch_union(graphs).to("cuda")
    got, rounds, maxc, _ = gc.gc_color_recolor_batch(u.offsets, u.idx, desc)
    got = got.cpu().numpy()
    base = 0
    for i, (g, d) in enumerate(zip(graphs, desc)):
        if g.n:
            off, idx = g.numpy()
            colors, _ = oracle.color(off, idx, d["X"], d["seed"])
            want, counts = oracle.recolor(off, idx, colors, d["perm"], d["iterations"], d["perm_seed"])
            assert np.array_equal(got[base:base + g.n], want), (name, i)
            assert maxc[i] == counts[-1]
        else:
            assert maxc[i] == 0 and rounds[i] == 0
        base += g.n
