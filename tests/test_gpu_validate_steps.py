"""gc_validate where its pass over the entries is cut: steps of 252 rows and
entries together (rows of 250 to 254 and around two steps, runs of empty
rows longer than a step), ids that do not start on a 16-byte boundary, and
colors that differ only above their low byte.  Counts are compared, equal,
with counts made on the CPU."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

DEGREES = {
    "steps": [250, 251, 252, 253, 254, 1, 0, 503, 504, 505, 2, 4097],
    "empty runs": [3] + [0] * 700 + [260] + [0] * 251 + [5] + [0] * 252,
    "ones": [1] * 1025,
    "one row": [9000] + [0] * 9,
    "no entries": [0] * 600,
}


def _expected(off, idx, colors):
    own = np.repeat(np.arange(len(off) - 1), np.diff(off))
    same = colors[own] == colors[idx]
    bad = np.zeros(len(off) - 1, bool)
    bad[own[same]] = True
    bad |= colors < 1
    return dict(n_conflicts=int(same.sum()), n_uncolored=int((colors < 1).sum()),
                max_color=max(0, int(colors.max())), n_distinct=len(np.unique(colors[colors >= 1])),
                first_bad_vertex=int(np.flatnonzero(bad)[0]) if bad.any() else -1)


@pytest.mark.parametrize("name", list(DEGREES))
@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("colors", ["many", "bytes", "one", "few bad"])
def test_counts(name, shift, colors):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(len(name) + 10 * shift)
    deg = np.array(DEGREES[name])
    n = len(deg)
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    idx = rng.integers(0, n, off[-1]).astype(np.int32)
    c = {"many": rng.integers(1, 70000, n),
         "bytes": 7 + 256 * rng.integers(0, 300, n),
         "one": np.full(n, 5),
         "few bad": np.arange(1, n + 1)}[colors].astype(np.int32)
    if colors == "few bad":  # in order, one vertex without a color
        idx = np.where(idx == np.repeat(np.arange(n), deg), (idx + 1) % n, idx).astype(np.int32)
        c[n // 2] = -4
    buf = torch.empty(off[-1] + shift, dtype=torch.int32, device="cuda")
    buf[shift:] = torch.from_numpy(idx)
    got = gc.gc_validate(torch.from_numpy(off).cuda(), buf[shift:], torch.from_numpy(c).cuda())
    assert {k: got[k] for k in _expected(off, idx, c)} == _expected(off, idx, c)


def test_an_id_out_of_range_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    off = torch.tensor([0] + [252 * (i + 1) for i in range(40)], dtype=torch.int64)
    idx = torch.zeros(252 * 40, dtype=torch.int32)
    colors = torch.arange(1, 41, dtype=torch.int32)
    for at in (0, 251, 252, 5000, 252 * 40 - 1):
        for bad in (-1, 40):
            ids = idx.clone()
            ids[at] = bad
            with pytest.raises(gc.GCError) as e:
                gc.gc_validate(off.cuda(), ids.cuda(), colors.cuda())
            assert e.value.name == "GC_ERR_BAD_GRAPH"
