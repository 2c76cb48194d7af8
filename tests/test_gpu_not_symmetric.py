"""A CSR that is not symmetric is outside the contract, but a call on one ends:
a neighbor that is not in the other's row does not push its color there, and
a round in which nobody wins turns the choices to the rows.  Before it did,
such a call ran its limit of n + 2 rounds."""
import time

import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    yield
    gc.gc_set_tuning()


def _rows(n, rows):
    off = torch.zeros(n + 1, dtype=torch.int64)
    for v, r in rows.items():
        off[v + 1] = len(r)
    idx = [torch.as_tensor(rows[v], dtype=torch.int32) for v in sorted(rows)]
    return off.cumsum(0).cuda(), torch.cat(idx).cuda()


def _path(n):
    return _rows(n, {v: [v + 1] for v in range(n - 1)})


def _star(n):  # the leaves know their hub, not it them
    return _rows(n, {v: [0] for v in range(1, n)})


def _out_star(n):
    return _rows(n, {0: list(range(1, n))})


def _random(n, seed, long_rows=()):
    rng = np.random.default_rng(seed)
    rows = {}
    for v in range(n):
        d = long_rows[v] if v < len(long_rows) else int(rng.integers(0, 9))
        r = np.unique(rng.integers(0, n, size=d))
        rows[v] = r[r != v]
    return _rows(n, rows)


GRAPHS = {
    "path": lambda: _path(100),
    "star": lambda: _star(100),
    "out-star": lambda: _out_star(100),
    "long-path": lambda: _path(40_000),
    "random": lambda: _random(5000, 1),
    "random-hubs": lambda: _random(5000, 2, (4000, 1500, 300, 70, 64)),
}


@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 2), ("RXF", 40), ("RXF", 80)])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_the_rounds_end(name, strategy, X):
    off, idx = GRAPHS[name]()
    n = off.numel() - 1
    deg = off[1:] - off[:-1]
    ref = None
    for seed in (1, 2, 3):
        for knobs in ({}, dict(spec_graph=0), dict(grid_blocks=2)):
            gc.gc_set_tuning(**knobs)
            colors, st = gc.gc_color(off, idx, strategy, X, seed)
            assert st["rounds"] < min(n, 60), knobs
            assert int(colors.min()) >= 1
            assert bool((colors <= deg + 192 + X).all())
            if not knobs:
                ref = colors
            # (a heavy row's list drops a fixed neighbor when it happens to see it, which makes
            # no difference on a symmetric CSR)
            if int(deg.max()) + X <= 64:
                assert torch.equal(colors, ref), knobs


@pytest.mark.parametrize("strategy,X", [("FF", 1), ("RXF", 3)])
def test_a_bad_id_in_a_large_graph_is_reported_at_once(strategy, X):
    """The entry is dropped, so its row and its neighbor's no longer match."""
    g = gg.erdos_renyi(1_000_000, 12.0, seed=3, device="cuda")
    gc.gc_color(g.offsets, g.idx, strategy, X, 1)
    idx = g.idx.clone()
    idx[1000::5000] = g.n
    torch.cuda.synchronize()
    t = time.perf_counter()
    with pytest.raises(gc.GCError) as e:
        gc.gc_color(g.offsets, idx, strategy, X, 1)
    assert e.value.name == "GC_ERR_BAD_GRAPH"
    assert time.perf_counter() - t < 0.5  # a coloring of it takes a millisecond


@pytest.mark.parametrize("name", ["random", "random-hubs", "path"])
def test_recoloring_stays_in_its_tables(name):
    """Several iterations on such a graph: colors, or an error, and the next call is right."""
    off, idx = GRAPHS[name]()
    for mode in (0, 1):
        gc.gc_set_tuning(recolor_mode=mode)
        for perm in ("RV", "NI", "RAND"):
            for strategy, X in (("FF", 1), ("RXF", 5)):
                try:
                    colors = gc.gc_color_recolor(off, idx, strategy, X, 3, perm, 5, 1)[0]
                    assert int(colors.min()) >= 1
                except gc.GCError as e:
                    assert e.name == "GC_ERR_IMPROPER_INPUT"
    gc.gc_set_tuning()
    g = gg.erdos_renyi(3000, 9.0, seed=5)
    val = gc.gc_color_recolor(g.offsets.cuda(), g.idx.cuda(), "FF", 1, 3, "RV", 3, 0, validate=True)[3]
    assert val["n_conflicts"] == 0 and val["n_uncolored"] == 0
