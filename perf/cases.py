"""The work that users of this library have it do, as cases that can be timed.

A case is one call of the Python binding with its graph: a coloring, a
coloring with recoloring iterations, the recoloring of a coloring at hand, a
validation, a batch of graphs in one CSR, or a call on host memory.  The
graphs are the library's workload families: G(n, p), 7- and 27-point box
meshes (natural or shuffled ids) and R-MAT with the Graph500 quadrant
probabilities or those of the RMAT-ER / RMAT-Good / RMAT-Bad classes, each
made on the GPU from the seed alone.

Every output is a whole number (colors, color counts, round and conflict
counts), so results are either equal or wrong.
"""
import math

import numpy as np
import torch

import paper_1407_6745_gb300 as gc

# (a, b, c) quadrant probabilities: Graph500, and the classes of the paper's Sec. 4.1
RMAT = {"graph500": (0.57, 0.19, 0.19), "er": (0.25, 0.25, 0.25), "good": (0.45, 0.15, 0.15),
        "bad": (0.55, 0.15, 0.15)}
PERMS = ("RV", "NI", "ND", "RAND", "ND-RAND%2^I")
INTS = ("rounds", "iterations", "max_color", "edges_examined", "conflicts")


def listed():
    return [
        # the smallest call: a graph of a thousand vertices, where launches and host work are all there is
        {"name": "er-1k-ff-rv2", "call": "color_recolor", "graph": "er", "n": 1000, "degree": 16.0,
         "strategy": "FF", "X": 1, "perm": "RV", "iterations": 2, "check": False},
        # a small sparse-matrix graph, colored, compacted and checked (the smallest benchmark workload)
        {"name": "er-10k-ff-rv2-check", "call": "color_recolor", "graph": "er", "n": 10_000, "degree": 16.0,
         "strategy": "FF", "X": 1, "perm": "RV", "iterations": 2, "check": True},
        # the "speed" preset: First Fit alone, on a mid-size graph without locality
        {"name": "er-1m-speed", "call": "color", "graph": "er", "n": 1_000_000, "degree": 24.0,
         "strategy": "FF", "X": 1},
        # the "quality" preset (Random-5 Fit + 1 ND iteration) on a box mesh in its natural order, odd sides
        {"name": "st7-odd-quality", "call": "color_recolor", "graph": "mesh", "x": 97, "y": 101, "z": 103,
         "points": 7, "shuffled": False, "strategy": "RXF", "X": 5, "perm": "ND", "iterations": 1,
         "check": False},
        # a finite-element mesh with shuffled ids, ten NI iterations, checked (the mesh benchmark workload)
        {"name": "st27-128-rx8-ni10", "call": "color_recolor", "graph": "mesh", "x": 128, "y": 128, "z": 128,
         "points": 27, "shuffled": True, "strategy": "RXF", "X": 8, "perm": "NI", "iterations": 10,
         "check": True},
        # one leg of the headline workload, the largest call: skewed degrees, hubs of 400 K entries
        {"name": "rmat24-ff-rand20", "call": "color_recolor", "graph": "rmat", "kind": "graph500", "scale": 24,
         "factor": 16, "strategy": "FF", "X": 1, "perm": "RAND", "iterations": 20, "check": True},
        # the headline's other strategy at a quarter of the size
        {"name": "rmat22-rx4-rand20", "call": "color_recolor", "graph": "rmat", "kind": "graph500", "scale": 22,
         "factor": 16, "strategy": "RXF", "X": 4, "perm": "RAND", "iterations": 20, "check": False},
        # the paper's most skewed class, First Fit and ten ND iterations, its own setting
        {"name": "rmatbad22-ff-nd10", "call": "color_recolor", "graph": "rmat", "kind": "bad", "scale": 22,
         "factor": 8, "strategy": "FF", "X": 1, "perm": "ND", "iterations": 10, "check": False},
        # a coloring at hand (read from a checkpoint, say) recolored further: the input is checked first
        {"name": "rmat18-recolor-rv5", "call": "recolor", "graph": "rmat", "kind": "graph500", "scale": 18,
         "factor": 16, "strategy": "FF", "X": 1, "perm": "RV", "iterations": 5},
        # a coloring checked after its graph was edited: one vertex in a thousand may have become wrong
        {"name": "rmat22-validate", "call": "validate", "graph": "rmat", "kind": "graph500", "scale": 22,
         "factor": 16, "strategy": "FF", "X": 1},
        # many independent graphs in one call, from a thousand vertices to a hundred thousand
        {"name": "batch-512", "call": "batch", "graph": "batch", "count": 512, "n_lo": 1000, "n_hi": 100_000,
         "sizes": 6, "X": 4, "perm": "RV", "iterations": 5},
        # a graph in pinned host memory, uploaded, colored and brought back by one call
        {"name": "rmat20-host-ff-rand5", "call": "host", "graph": "rmat", "kind": "graph500", "scale": 20,
         "factor": 16, "strategy": "FF", "X": 1, "perm": "RAND", "iterations": 5, "check": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(("color_recolor", "color_recolor", "color_recolor", "color", "recolor", "validate",
                       "batch", "host"))
    if call == "batch":
        return {"call": call, "graph": "batch", "count": _log_int(rng, 16, 512), "n_lo": 1000,
                "n_hi": _log_int(rng, 10_000, 100_000), "sizes": rng.randint(0, 9999),
                "X": rng.randint(1, 8), "perm": rng.choice(PERMS), "iterations": rng.randint(0, 6)}
    graph = rng.choice(("er", "mesh", "rmat"))
    case = {"call": call, "graph": graph}
    if graph == "er":
        case |= {"n": _log_int(rng, 1000, 1_000_000), "degree": round(rng.uniform(8.0, 32.0), 2)}
    elif graph == "mesh":
        case |= {"x": _log_int(rng, 16, 128), "y": _log_int(rng, 16, 128), "z": _log_int(rng, 16, 128),
                 "points": rng.choice((7, 27)), "shuffled": rng.random() < 0.5}
    else:
        kind = rng.choice(tuple(RMAT))
        case |= {"kind": kind, "scale": rng.randint(14, 21 if call == "host" else 23),
                 "factor": rng.randint(8, 16) if kind == "graph500" else 8}
    x = rng.choice((1, rng.randint(2, 10)))
    case |= {"strategy": "FF" if x == 1 else "RXF", "X": x}
    if call in ("color_recolor", "recolor", "host"):
        case |= {"perm": rng.choice(PERMS), "iterations": rng.randint(1, 20)}
    if call in ("color_recolor", "host"):
        case["check"] = rng.random() < 0.5
    return case


# ---------------------------------------------------------------------------
# Graphs: symmetric CSR, no loops, no duplicates, rows sorted
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csr(n, src, dst, both):
    key = torch.cat([src * n + dst, dst * n + src]) if both else src * n + dst
    key = torch.unique_consecutive(torch.sort(key).values)
    row = torch.div(key, n, rounding_mode="floor")
    idx = (key - row * n).to(torch.int32)
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=offsets[1:])
    return offsets, idx


def _er(n, degree, seed):
    m = int(n * degree / 2)
    ends = torch.randint(0, n, (2, m), generator=_gen(seed), device="cuda")
    ends = ends[:, ends[0] != ends[1]]
    return _csr(n, ends[0], ends[1], True)


def _mesh_edges(v, x, y, z, sx, sy, sz, points):
    """Entries (source, target) of box meshes: vertex v at (x, y, z) of a box of sides (sx, sy, sz)."""
    srcs, dsts = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if (dx, dy, dz) == (0, 0, 0) or (points == 7 and abs(dx) + abs(dy) + abs(dz) != 1):
                    continue
                ok = ((x + dx >= 0) & (x + dx < sx) & (y + dy >= 0) & (y + dy < sy)
                      & (z + dz >= 0) & (z + dz < sz))
                srcs.append(v[ok])
                dsts.append((v + dx + sx * (dy + sy * dz))[ok])
    return torch.cat(srcs), torch.cat(dsts)


def _mesh(case, seed):
    sx, sy, sz = case["x"], case["y"], case["z"]
    n = sx * sy * sz
    v = torch.arange(n, device="cuda")
    src, dst = _mesh_edges(v, v % sx, (v // sx) % sy, v // (sx * sy), sx, sy, sz, case["points"])
    if case["shuffled"]:
        perm = torch.randperm(n, generator=_gen(seed), device="cuda")
        src, dst = perm[src], perm[dst]
    return _csr(n, src, dst, False)


def _rmat(case, seed):
    a, b, c = RMAT[case["kind"]]
    n, m, gen = 1 << case["scale"], case["factor"] << case["scale"], _gen(seed)
    srcs, dsts = [], []
    for start in range(0, m, 1 << 26):
        cnt = min(1 << 26, m - start)
        u = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        w = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        for _ in range(case["scale"]):
            r = torch.rand(cnt, generator=gen, device="cuda")
            down = r >= a + b
            right = torch.where(down, r >= a + b + c, r >= a)
            u = 2 * u + down
            w = 2 * w + right
        keep = u != w
        srcs.append(u[keep])
        dsts.append(w[keep])
    return _csr(n, torch.cat(srcs), torch.cat(dsts), True)


def _batch(case, seed):
    """Half G(n, p) of mean degree U[8, 32], half 2D 5-point or 3D 7-point grids in natural order; the
    sizes are the case's own, the edges and the graphs' seeds come from the seed."""
    rng = np.random.default_rng(case["sizes"])
    sizes, ers, meshes, base = [], [], [], 0
    for i in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        if i % 2 == 0:
            ers.append((base, n, int(n * rng.uniform(8.0, 32.0) / 2)))
        else:
            flat = rng.random() < 0.5
            side = int(round(n ** (1 / 2 if flat else 1 / 3)))
            meshes.append((base, side, side, 1 if flat else side))
            n = side * side * (1 if flat else side)
        sizes.append(n)
        base += n
    srcs, dsts = [], []

    def spread(rows, counts):
        rows = torch.tensor(rows, device="cuda")
        at = torch.repeat_interleave(torch.arange(len(rows), device="cuda"), torch.tensor(counts, device="cuda"))
        return rows[at].T

    if ers:
        first, n, _ = spread(ers, [m for _, _, m in ers])
        r = torch.rand((2, first.numel()), generator=_gen(seed), device="cuda", dtype=torch.float64)
        u, w = ((r * n).to(torch.int64) + first).unbind(0)
        keep = u != w
        srcs += [u[keep], w[keep]]
        dsts += [w[keep], u[keep]]
    if meshes:
        counts = [x * y * z for _, x, y, z in meshes]
        first, sx, sy, sz = spread(meshes, counts)
        start = torch.tensor(np.cumsum([0] + counts[:-1]), device="cuda")
        local = torch.arange(first.numel(), device="cuda") - torch.repeat_interleave(
            start, torch.tensor(counts, device="cuda"))
        s, d = _mesh_edges(first + local, local % sx, (local // sx) % sy, local // (sx * sy), sx, sy, sz, 7)
        srcs.append(s)
        dsts.append(d)
    off, idx = _csr(base, torch.cat(srcs), torch.cat(dsts), False)
    graphs = [{"n": n, "seed": seed + 1000 + i, "X": case["X"], "perm": case["perm"],
               "iterations": case["iterations"], "perm_seed": seed + i} for i, n in enumerate(sizes)]
    return off, idx, graphs


# ---------------------------------------------------------------------------

def prepare(case, seed):
    state = {"case": case, "seed": seed + 7, "perm_seed": seed + 5}
    if case["graph"] == "batch":
        state["offsets"], state["idx"], state["graphs"] = _batch(case, seed)
        return state
    if case["graph"] == "er":
        off, idx = _er(case["n"], case["degree"], seed)
    elif case["graph"] == "mesh":
        off, idx = _mesh(case, seed)
    else:
        off, idx = _rmat(case, seed)
    if case["call"] in ("recolor", "validate"):
        state["colors"], _ = gc.gc_color(off, idx, case["strategy"], case["X"], state["seed"])
    if case["call"] == "validate":
        n = off.numel() - 1
        at, other = torch.randint(0, n, (2, n // 1000 + 8), generator=_gen(seed), device="cuda")
        state["colors"][at] = state["colors"][other]
    if case["call"] == "host":
        off, idx = off.cpu().pin_memory(), idx.cpu().pin_memory()
        state["out"] = torch.empty(off.numel() - 1, dtype=torch.int32).pin_memory()
    state["offsets"], state["idx"] = off, idx
    return state


def run(state):
    c, off, idx = state["case"], state["offsets"], state["idx"]
    if c["call"] == "batch":
        colors, rounds, max_color, st = gc.gc_color_recolor_batch(off, idx, state["graphs"])
        return {"colors": colors, "rounds": np.array(rounds), "max_color": np.array(max_color),
                "edges_examined": st["edges_examined"]}
    if c["call"] == "color":
        colors, st = gc.gc_color(off, idx, c["strategy"], c["X"], state["seed"])
        return {"colors": colors, "stats": {k: st[k] for k in INTS}}
    if c["call"] == "recolor":
        colors, counts, st = gc.gc_recolor(off, idx, state["colors"], c["perm"], c["iterations"],
                                           state["perm_seed"])
        return {"colors": colors, "counts": np.array(counts), "stats": {k: st[k] for k in INTS}}
    if c["call"] == "validate":
        return gc.gc_validate(off, idx, state["colors"])
    colors, counts, st, check = gc.gc_color_recolor(
        off, idx, c["strategy"], c["X"], state["seed"], c["perm"], c["iterations"], state["perm_seed"],
        out=state.get("out"), validate=c["check"])
    return {"colors": colors, "counts": np.array(counts), "stats": {k: st[k] for k in INTS},
            "check": check or {}}


def _size(case):
    """(vertices, adjacency entries) that the case's graph is expected to have."""
    if case["graph"] == "er":
        return case["n"], case["n"] * case["degree"]
    if case["graph"] == "mesh":
        x, y, z = case["x"], case["y"], case["z"]
        n = x * y * z
        if case["points"] == 27:
            return n, (3 * x - 2) * (3 * y - 2) * (3 * z - 2) - n
        return n, 2 * (3 * n - x * y - y * z - x * z)
    if case["graph"] == "batch":  # log-uniform sizes; mean degree 20 (G(n, p)) and about 5 (grids)
        lo, hi = case["n_lo"], case["n_hi"]
        n = case["count"] * (hi - lo) / math.log(hi / lo) if hi > lo else case["count"] * lo
        return n, 12.5 * n
    n = 1 << case["scale"]  # nearly all generated edges are distinct, fewer with the Graph500 skew
    return n, 2 * case["factor"] * n * (0.93 if case["kind"] == "graph500" else 0.99)


def work(case):
    """Each step (the coloring, every recoloring iteration, the validation) depends on the whole result
    of the one before it, so each reads the graph once, reads the colors it starts from and writes its own."""
    n, nnz = _size(case)
    graph = 8 * (n + 1) + 4 * nnz
    color, recolor, check = graph + 4 * n, graph + 8 * n, graph + 4 * n
    if case["call"] == "validate":
        total = check
    elif case["call"] == "color":
        total = color
    elif case["call"] == "recolor":
        total = check + case["iterations"] * recolor
    else:
        total = color + case["iterations"] * recolor + (check if case.get("check") else 0)
    return {"bytes": float(total), "flops": 0.0}


def exact(case, seed):
    """No output has a value in 64 bits to be near to: all are whole numbers and have to be equal."""
    return None
