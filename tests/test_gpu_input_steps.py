"""The check of a recoloring input (gc_recolor with no iterations: the check
and a copy) where its pass over the entries is cut: rows around one and two
steps of 252 rows and entries, rows inside which whole steps lie, rows around
the 128 steps that a thread writes the starts of itself, ids that do not
start on a 16-byte boundary; all colors share their low byte."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")

DEGREES = {
    "steps": [250, 251, 252, 253, 254, 1, 0, 503, 504, 505, 2, 4097],
    "long rows": [3, 128 * 252 - 2, 128 * 252 - 1, 0, 128 * 252, 128 * 252 + 253, 1, 200_000, 5],
    "many long rows": [33_000 + i for i in range(40)] + [1] * 70,
}


@pytest.fixture(params=[(k, s) for k in DEGREES for s in (0, 1, 3)], ids=lambda p: f"{p[0]}-{p[1]}")
def case(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    name, shift = request.param
    deg = np.array(DEGREES[name])
    n = len(deg)
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    own = np.repeat(np.arange(n), deg)
    idx = (own + np.random.default_rng(shift).integers(1, n, off[-1])) % n  # never the row itself
    colors = 7 + 256 * np.random.default_rng(1).permutation(n)

    def check(idx=idx, colors=colors):
        buf = torch.empty(off[-1] + shift, dtype=torch.int32, device="cuda")
        buf[shift:] = torch.from_numpy(idx.astype(np.int32))
        c = torch.from_numpy(colors.astype(np.int32)).cuda()
        d_off = torch.from_numpy(off).cuda()
        try:
            out, counts, _ = gc.gc_recolor(d_off, buf[shift:], c, "RV", 0)
            assert torch.equal(out, c) and counts == [int(colors.max())]
            status = "GC_OK"
        except gc.GCError as e:
            status = e.name
        if colors.min() >= 1 and status != "GC_ERR_BAD_GRAPH":  # the validation agrees
            assert (gc.gc_validate(d_off, buf[shift:], c)["n_conflicts"] == 0) == (status == "GC_OK")
        return status

    return off, own, idx, colors, check


def test_equal_low_bytes_are_proper(case):
    assert case[4]() == "GC_OK"


def test_one_bad_entry_or_color(case):
    off, own, idx, colors, check = case
    n, nnz = len(colors), int(off[-1])
    places = {0, 251, 252, 253, 503, 504, nnz - 1, nnz // 2} | {int(e) for e in off[1:-1] if e < nnz} \
        | {int(e) - 1 for e in off[1:] if e > 0}
    for e in sorted(places)[:60]:
        bad = idx.copy()
        bad[e] = own[e]  # the row's own color
        assert check(idx=bad) == "GC_ERR_IMPROPER_INPUT", e
        bad[e] = n
        assert check(idx=bad) == "GC_ERR_BAD_GRAPH", e
        c = colors.copy()  # an id is not looked at in a row without a valid color
        c[own[e]] = 0
        assert check(idx=bad, colors=c) == "GC_ERR_IMPROPER_INPUT", e
