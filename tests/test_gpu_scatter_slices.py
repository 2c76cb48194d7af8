"""The recoloring's lists on both sides of 2^24 vertices, from where on a graph
without split rows is dealt out in slices: equal to the oracle."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")


@pytest.mark.parametrize("x,y", [(4096, 4096), (4097, 4096)])
def test_grids(x, y):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    g = gg.grid_2d(x, y, device="cuda")
    colors, _ = gc.gc_color(g.offsets, g.idx, "RXF", 4, 9)
    got, nc, st = gc.gc_recolor(g.offsets, g.idx, colors, "RAND", 1, 5)
    want, counts = oracle.recolor(g.offsets.cpu().numpy(), g.idx.cpu().numpy(), colors.cpu().numpy(), "RAND", 1, 5)
    assert np.array_equal(got.cpu().numpy(), want)
    assert nc == counts.tolist() and st["edges_examined"] == g.nnz
