"""Device memory of a census: a bipartite graph (no lists, no core) takes what
its adjacency entries need and little else."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Bytes per adjacency entry: the loaded entries 4; renamed 4; reverse slots 8; T 4; K4 8; C4 8; list and position
# offsets 16; sort keys 16 and digit counts 1.  Half a record (8) more is allowed for the per-vertex arrays, the counter
# scratch and the rounding of some forty allocations.
ENTRIES = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
torch.cuda.set_device(0)
import graphgen as gg
from paper_1610_09411_gb300 import escape as esc
g0 = gg.erdos_renyi(100, 0.1, 1)
esc.census(g0.row_ptr, g0.col, n=g0.n)
g = gg.complete_bipartite(900, 7200)
free, _ = torch.cuda.mem_get_info()
h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
c = esc.escape_census5(h)
per = (free - torch.cuda.mem_get_info()[0]) / g.nnz    # released buffers are kept, each was in use once
assert c["n3"][3] == 0 and c["n4"][3] == 900 * 899 // 2 * (7200 * 7199 // 2)
print("bytes per entry", per)
assert per <= 69 + 8
"""


def test_bytes_per_adjacency_entry():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", ENTRIES, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
