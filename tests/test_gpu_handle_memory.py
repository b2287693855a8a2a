"""Device memory of handles: what a freed handle of a large graph took goes back
to the device, and a handle holds little more than its graph needs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import torch
torch.cuda.set_device(0)
import graphgen as gg
from paper_1610_09411_gb300 import escape as esc
g0 = gg.erdos_renyi(100, 0.1, 1)
esc.census(g0.row_ptr, g0.col, n=g0.n)

def ring(n, d):
    v = np.arange(n)
    return gg.from_edges(n, np.repeat(v, d // 2), (v[:, None] + np.arange(1, d // 2 + 1)).ravel() % n)

def free():
    return torch.cuda.mem_get_info()[0]

MB = 1 << 20
"""
SCRIPTS = {
    # rows of 80 MB, entries of 160 MB
    "loaded": """
g = ring(10000000, 4)
before = free()
h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
assert before - free() >= 220 * MB
esc.escape_free(h)
assert before - free() <= 90 * MB, (before - free()) / MB
""",
    # T 160, C4 320, K4 320, renamed entries 160, reverse slots 320 and the loaded entries 160 MB
    "elements": """
g = ring(10000000, 4)
h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
esc.escape_set_options(h, keep_per_element=True)
esc.escape_census5(h)
held = free()
esc.escape_free(h)
assert free() - held >= 1360 * MB, (free() - held) / MB
""",
    # raw entries of twice the size are not part of the handle
    "normalised": """
g = ring(10000000, 4)
before = free()
h = esc.escape_load_csr(g.n, g.row_ptr, g.col, flags=esc.ESCAPE_NORMALIZE)
held = free()
esc.escape_free(h)
assert free() - held >= 152 * MB, (free() - held) / MB
""",
    # a kept buffer of 60 MB is not taken for 32 MB of entries
    "tight": """
a, b = ring(250000, 60), ring(250000, 32)
esc.escape_free(esc.escape_load_csr(a.n, a.row_ptr, a.col))
before = free()
h = esc.escape_load_csr(b.n, b.row_ptr, b.col)
assert before - free() >= 28 * MB, (before - free()) / MB
esc.escape_free(h)
""",
}


@pytest.mark.parametrize("name", list(SCRIPTS))
def test_memory_of_handles(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", HEAD + SCRIPTS[name], ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
