"""The two layouts of the color words (color and priority in one 8-byte word
up to 15 * 2^18 vertices, arrays of their own beyond), each in every form that
the rounds can be run in, bit-exact against the oracle, with statistics."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

WIDE_MAX = 15 << 18
FORMS = [dict(), dict(spec_graph=0), dict(grid_blocks=5), dict(g2_max_deg=0), dict(g2_max_deg=4, g4_max_deg=8, g8_max_deg=16,
                                                                                  g16_max_deg=32)]


@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 3)])
@pytest.mark.parametrize("hubs", [[], [3000, 1100, 300, 200, 64, 63]])
@pytest.mark.parametrize("n", [WIDE_MAX, WIDE_MAX + 1])
def test_every_form_of_both_layouts(n, hubs, strategy, X):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = gg.hubs(hubs, n - len(hubs), seed=2, device="cuda")
    assert g.n == n
    want, stats = oracle.color(*g.numpy(), X, 5)
    want = torch.from_numpy(np.ascontiguousarray(want)).cuda()
    room = torch.empty(g.nnz + 1, dtype=torch.int32, device="cuda")
    room[1:] = g.idx
    try:
        for knobs in FORMS:
            for idx in (g.idx, room[1:]):  # 16-byte aligned, and not
                gc.gc_set_tuning(**knobs)
                got, st = gc.gc_color(g.offsets, idx, strategy, X, 5)
                assert torch.equal(got, want), knobs
                assert all(st[k] == stats[k] for k in ("rounds", "max_color", "edges_examined", "conflicts")), knobs
                gc.gc_set_tuning()
    finally:
        gc.gc_set_tuning()
