"""Recoloring inputs with the largest colors that are taken, 2^28 - 1 and
2^28: the (class, degree bucket) tables over them stay within 32-bit indices.
An iteration depends on the order of the classes and on their sizes only, so
the result is that of the same coloring with its last class at a small color."""
import re
from pathlib import Path

import pytest
import torch

import graphgen as gg

gc = pytest.importorskip("paper_1407_6745_gb300")

MAX_COLOR = 1 << 28


def test_class_tables_fit_32_bit_indices():
    src = (Path(gc.__file__).parent / "csrc" / "gc_recolor.cu").read_text()
    buckets = int(re.search(r"constexpr int kRcNB = (\d+);", src).group(1))
    shift = int(re.search(r"constexpr int32_t kMaxInputColor = 1 << (\d+);", src).group(1))
    assert 1 << shift == MAX_COLOR
    assert (MAX_COLOR + 1) * buckets < 1 << 31


@pytest.mark.gpu
@pytest.mark.parametrize("top", [MAX_COLOR - 1, MAX_COLOR])
def test_largest_input_colors(top):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("the class tables take about 50 GB")
    gc.gc_set_tuning()
    g = gg.hubs([100, 300], 3000, seed=4)
    off, idx = g.offsets.cuda(), g.idx.cuda()
    small, _ = gc.gc_color(off, idx, "RXF", 6, 2)
    big = torch.where(small == small.max(), top, small)
    for perm in ("RV", "RAND"):
        want, counts, _ = gc.gc_recolor(off, idx, small, perm, 2, 9)
        got, big_counts, _ = gc.gc_recolor(off, idx, big, perm, 2, 9)
        assert torch.equal(got, want), perm
        assert big_counts == [top] + counts[1:], perm
    want = gc.gc_recolor_async(off, idx, small, "RV", 1, 9)
    got = gc.gc_recolor_async(off, idx, big, "RV", 1, 9)
    assert torch.equal(got[0], want[0]) and got[1][1:] == want[1][1:]


@pytest.mark.gpu
@pytest.mark.parametrize("knobs", [dict(g4_max_deg=4, g8_max_deg=8, g16_max_deg=16, g2_max_deg=0, rc_g2_max_deg=0),
                                   dict(g4_max_deg=0, g8_max_deg=0, g16_max_deg=0, g2_max_deg=0, rc_g2_max_deg=0),
                                   dict(rc_warp_max_deg=0), dict(rc_warp_max_deg=5000)])
def test_warp_rows_on_either_side_of_64_entries(knobs):
    """A warp's row keeps its colors in 64 register bits up to 63 entries, in a bitmap beyond."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = gg.hubs([1, 4, 5, 8, 9, 16, 17, 31, 33, 47, 62, 63, 64, 65, 66, 200, 512, 513, 3000], 6000, seed=5)
    off, idx = g.offsets.cuda(), g.idx.cuda()
    gc.gc_set_tuning()
    start, _ = gc.gc_color(off, idx, "RXF", 70, 3)
    want, counts, _ = gc.gc_recolor(off, idx, start, "NI", 3, 1)
    try:
        for mode in (0, 1):
            gc.gc_set_tuning(recolor_mode=mode, **knobs)
            got, c, _ = gc.gc_recolor(off, idx, start, "NI", 3, 1)
            assert torch.equal(got, want) and c == counts
    finally:
        gc.gc_set_tuning()
