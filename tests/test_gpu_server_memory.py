"""The server's estimate of a request's device memory covers what the request
takes: graphs with heavy rows (lists of their neighbors, bitmaps, queues), split
rows and none, each served alone by a fresh process, whose free memory before
and after gives what the library's pool had to reserve."""
import json
import subprocess
import sys
from pathlib import Path

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parents[1]
SLACK = 192 << 20  # kernels loaded meanwhile, and the pool's own rounding

SERVE = """
import json, sys, torch
sys.path.insert(0, %r)
import graphgen as gg
import paper_1407_6745_gb300 as gc
gc.load()
g = %s
off, idx = g.offsets.cpu(), g.idx.cpu()
w = gg.erdos_renyi(3000, 80.0, seed=1).to("cuda")
gc.gc_color_recolor(w.offsets, w.idx, "FF", 1, 1, "RV", 2)
del g
torch.cuda.synchronize()
torch.cuda.empty_cache()
free = torch.cuda.mem_get_info()[0]
with gc.gc_server_create(100 << 30, 4, 1) as srv:
    gc.gc_server_wait(srv, gc.gc_server_submit(srv, off, idx, %r, %d, 1, "RV", 3))
    peak = gc.gc_server_stats(srv)["bytes_peak"]
    print(json.dumps({"taken": free - torch.cuda.mem_get_info()[0], "estimate": peak}))
"""


@pytest.mark.parametrize("graph,strategy,X", [
    ("gg.erdos_renyi(40_000, 2000.0, seed=3, device='cuda')", "FF", 1),        # every row heavy and split
    ("gg.erdos_renyi(600_000, 100.0, seed=3, device='cuda')", "FF", 1),        # every row heavy, none split
    ("gg.erdos_renyi(6_000_000, 8.0, seed=3, device='cuda')", "RXF", 70),      # every row heavy and short
    ("gg.erdos_renyi(6_000_000, 16.0, seed=3, device='cuda')", "FF", 1),       # none
    ("gg.rmat(21, 16, 0.57, 0.19, 0.19, seed=4, device='cuda')", "FF", 1),
])
def test_estimate_covers_the_request(graph, strategy, X):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = subprocess.run([sys.executable, "-c", SERVE % (str(ROOT), graph, strategy, X)], capture_output=True,
                         text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    r = json.loads(out.stdout.strip().splitlines()[-1])
    assert r["taken"] <= r["estimate"] + SLACK, r
    assert r["taken"] > 200 << 20, r  # (it has been measured at all)
