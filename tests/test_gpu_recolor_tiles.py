"""The recoloring kernel's tiles where their geometry changes, bit-exact
against the oracle: rows at the edges of the 1-, 2- and 4-lane buckets and of
what a lane takes at once, rows at the end of the id array, ids that are not
16-byte aligned, more colors than one shared bitmap window holds, and split
rows with more in-flight neighbors than their list of left ones takes."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

gc = pytest.importorskip("paper_1407_6745_gb300")


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gc.gc_set_tuning()
    yield
    gc.gc_set_tuning()


def _multipartite(parts, size):
    n = parts * size
    part = torch.arange(n) // size
    src, dst = torch.nonzero(part[:, None] != part[None, :], as_tuple=True)
    return gg.csr_from_edges(n, src, dst, symmetrize=False, name=f"K_{parts}x{size}")


def _check(g, X, perm, iterations, seed=5, aligned=True):
    off, idx = g.numpy()
    colors, _ = oracle.color(off, idx, X, 3)
    want, counts = oracle.recolor(off, idx, colors, perm, iterations, seed)
    d_off, d_idx = g.offsets.cuda(), g.idx.cuda()
    if not aligned:
        room = torch.empty(g.nnz + 1, dtype=torch.int32, device="cuda")
        room[1:] = d_idx
        d_idx = room[1:]
    for mode in (0, 1):
        gc.gc_set_tuning(recolor_mode=mode)
        got, nc, st = gc.gc_recolor(d_off, d_idx, torch.from_numpy(colors).cuda(), perm, iterations, seed)
        assert np.array_equal(got.cpu().numpy(), want), (g.name, perm, mode)
        assert nc == counts.tolist()
        assert st["edges_examined"] == iterations * g.nnz


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("perm", ["RV", "RAND"])
def test_row_lengths(perm, aligned):
    degrees = [1, 2, 4, 7, 8, 9, 15, 16, 17, 31, 32, 33, 36, 37, 62, 63, 64, 65, 255, 256, 257, 315, 316,
               317, 511, 512, 513, 768, 769] * 3
    _check(gg.hubs(degrees, 5000, seed=4), 6, perm, 3, aligned=aligned)


@pytest.mark.parametrize("n,degree", [(33, 2.0), (257, 6.0), (4097, 9.0), (9999, 17.0)])
def test_odd_sizes(n, degree):
    _check(gg.erdos_renyi(n, degree, seed=n), 3, "NI", 3)


def test_more_colors_than_a_bitmap_window():
    _check(gg.complete(2100), 1, "RAND", 2)


@pytest.mark.parametrize("parts,size", [(5, 300), (3, 600)])
def test_more_in_flight_neighbors_than_the_list_takes(parts, size):
    _check(_multipartite(parts, size), 4, "RAND", 3)
