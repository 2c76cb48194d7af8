"""Random-X Fit where round 0 pushes nothing and its losers gather their marks:
on either layout of the color words, with light rows only, with heavy rows
around the piece length, with every row heavy, and in a batch; bit-exact
against the oracle, with statistics, in every form of the rounds."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

WIDE_MAX = 15 << 18
HUBS = [63, 64, 65, 127, 128, 129, 255, 256, 257, 1025, 30000]
FORMS = [dict(), dict(spec_graph=0), dict(grid_blocks=5)]


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    yield
    gc.gc_set_tuning()


def _launches():
    return gc.gc_profile_read().get("k_late_marks", (0, 0.0))[0]


def _check(g, X, seed):
    """Colors and statistics in every form, and that the marks were gathered."""
    want, stats = oracle.color(*g.numpy(), X, seed)
    want = torch.from_numpy(np.ascontiguousarray(want)).cuda()
    room = torch.empty(g.nnz + 1, dtype=torch.int32, device="cuda")
    room[1:] = g.idx
    for knobs in FORMS:
        for idx in (g.idx, room[1:]):
            gc.gc_set_tuning(**knobs)
            gc.gc_profile_enable(True)
            try:
                got, st = gc.gc_color(g.offsets, idx, "RXF", X, seed)
                launches = _launches()
            finally:
                gc.gc_profile_enable(False)
                gc.gc_set_tuning()
            assert launches == 1, knobs
            assert torch.equal(got, want), knobs
            assert all(st[k] == stats[k] for k in ("rounds", "max_color", "edges_examined", "conflicts")), knobs


@pytest.mark.parametrize("X", [40, 62, 100])
def test_shared_words(X):
    """Some rows heavy, nearly all, all of them (empty ones too)."""
    g = gg.erdos_renyi(300_000, 12.0, seed=4, device="cuda")
    h = gg.hubs(HUBS, 40_000, seed=3, device="cuda")
    _check(gg.batch_union([g, h, gg.empty(5).to("cuda")]), X, 7)


@pytest.mark.parametrize("X", [4, 70])
@pytest.mark.parametrize("hubs", [[], HUBS])
def test_separate_words(hubs, X):
    _check(gg.hubs(hubs, WIDE_MAX + 1 - len(hubs), seed=2, device="cuda"), X, 5)


def test_separate_words_of_many_vertices():
    """Light rows only, two thirds of the entries in losers."""
    _check(gg.erdos_renyi((9 << 20) + 5, 6.0, seed=6, device="cuda"), 2, 9)


def test_batch_of_different_X():
    graphs = [gg.erdos_renyi(n, d, seed=s) for s, (n, d) in enumerate([(120_000, 20.0), (300, 5.0), (90_000, 9.0), (1, 0.0)])]
    graphs.append(gg.hubs(HUBS, 35_000, seed=8))
    desc = [dict(n=g.n, seed=3 + i, X=x) for i, (g, x) in enumerate(zip(graphs, (60, 1, 90, 2, 45)))]
    u = gg.batch_union(graphs).to("cuda")
    gc.gc_profile_enable(True)
    try:
        colors, rounds, maxc, _ = gc.gc_color_batch(u.offsets, u.idx, desc)
        assert _launches() == 1
    finally:
        gc.gc_profile_enable(False)
    at = 0
    for g, d, r, m in zip(graphs, desc, rounds, maxc):
        want, stats = oracle.color(*g.numpy(), d["X"], d["seed"])
        assert np.array_equal(colors[at:at + g.n].cpu().numpy(), want)
        assert (r, m) == (stats["rounds"], stats["max_color"])
        at += g.n
