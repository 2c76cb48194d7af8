"""The speculative rounds where their geometry changes, bit-exact against the
oracle (colors and statistics): rows at the edges of the lane buckets, of the
shared-memory stage of a row, of the row and list pieces and of the list head;
ids that are not 16-byte aligned; rounds driven one launch at a time; small
and odd grids; and the two layouts of the color words on either side of the
vertex count where they change."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

DEGREES = [0, 1, 3, 4, 5, 7, 8, 9, 28, 31, 32, 33, 34, 35, 36, 37, 59, 60, 62, 63, 64, 65, 127, 128, 129, 255, 256,
           511, 512, 513, 1023, 1024, 1025, 1500, 2047, 2049, 4100]


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    yield
    gc.gc_set_tuning()


def _check(g, strategy, X, seed, aligned=True, off=None, idx=None):
    off, idx = off if off is not None else g.offsets.cuda(), idx if idx is not None else g.idx.cuda()
    want, stats = oracle.color(*g.numpy(), X, seed)
    if not aligned:
        room = torch.empty(g.nnz + 1, dtype=torch.int32, device="cuda")
        room[1:] = idx
        idx = room[1:]
    got, st = gc.gc_color(off, idx, strategy, X, seed)
    assert np.array_equal(got.cpu().numpy(), want), g.name
    for k in ("rounds", "max_color", "edges_examined", "conflicts"):
        assert st[k] == stats[k], (g.name, k)


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("knobs", [{}, dict(spec_graph=0), dict(grid_blocks=3), dict(g2_max_deg=0),
                                   dict(g2_max_deg=64, g4_max_deg=64)])
@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 5), ("RXF", 70)])
def test_row_lengths(strategy, X, knobs, aligned):
    gc.gc_set_tuning(**knobs)
    _check(gg.hubs(DEGREES * 2, 5000, seed=6), strategy, X, 9, aligned)


@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 4)])
@pytest.mark.parametrize("n,degree", [(1, 0.0), (2, 0.5), (17, 4.0), (511, 9.0), (4099, 30.0), (9973, 55.0)])
def test_odd_sizes(n, degree, strategy, X):
    _check(gg.erdos_renyi(n, degree, seed=n + 1), strategy, X, 3)


@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 3)])
@pytest.mark.parametrize("hubs", [[], [3000, 200, 64]])
@pytest.mark.parametrize("n", [(10 << 20) - 1, (10 << 20) + 3])
def test_layouts_of_the_color_words(n, hubs, strategy, X):
    """Below and above the vertex count up to which color and priority share a word."""
    g = gg.hubs(hubs, n - len(hubs), seed=2, device="cuda")
    assert g.n == n
    _check(g, strategy, X, 5, off=g.offsets, idx=g.idx)


def test_a_dense_core_with_long_lists():
    """Hubs that are all neighbors of each other and of many light vertices: long lists, lost and won in every round."""
    rng = np.random.default_rng(3)
    core, n = 300, 20000
    src = [np.repeat(np.arange(core), core), np.repeat(np.arange(core), 4000)]
    dst = [np.tile(np.arange(core), core), rng.integers(core, n, size=core * 4000)]
    g = gg.csr_from_edges(n, torch.from_numpy(np.concatenate(src)), torch.from_numpy(np.concatenate(dst)),
                          name="core")
    for strategy, X in (("FF", 1), ("RXF", 6)):
        _check(g, strategy, X, 4)
