"""Estimates of the device memory of a census: the serving loop's footprint and
the batch's chunk estimate charge the dense core, and what a census takes on
the GPU stays below them."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import graphgen as gg
from paper_1610_09411_gb300 import build as pb
from paper_1610_09411_gb300.serve import footprint_bytes, triangle_bound

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _footprint(g):
    deg = g.degrees()
    return footprint_bytes(g.n, g.m, triangle_bound(g.row_ptr, g.col), int(deg.max()))


def _regular(n, d):
    """Circulant graph: every vertex joined to the d / 2 next ones."""
    v = np.arange(n)
    return gg.from_edges(n, np.repeat(v, d // 2), (v[:, None] + np.arange(1, d // 2 + 1)).ravel() % n, f"ring{n}_{d}")


def test_footprint_charges_the_core():
    for n in (4000, 33000, 60000):
        g = _regular(n, 48)
        assert _footprint(g) >= 2 * n * n + 48 * n * 2          # W, and the entries at least
    thin, thick = _regular(33000, 46), _regular(33000, 48)     # no core vertex: no W
    assert _footprint(thin) < 2 * 33000 ** 2 < _footprint(thick)
    # counts of 32 bits; W beyond its limit: no core
    assert footprint_bytes(70000, 200000, 0, 65536, core_vertices=20000) - \
        footprint_bytes(70000, 200000, 0, 65536, core_vertices=0) >= 4 * 20000 ** 2
    assert footprint_bytes(10 ** 6, 10 ** 8, 0, 1000, core_vertices=200000) == \
        footprint_bytes(10 ** 6, 10 ** 8, 0, 1000, core_vertices=0)


@pytest.fixture(scope="module")
def estimate(tmp_path_factory):
    d = tmp_path_factory.mktemp("estimate")
    src, so = str(d / "e.cpp"), str(d / "e.so")
    with open(src, "w") as f:
        f.write('#include "estimate.h"\n'
                'extern "C" double estimate(const int64_t* rp, const int64_t* voff, int graphs, int sms) {\n'
                '  esc::ChunkEstimate e;\n'
                '  for (int k = 0; k < graphs; ++k) e.add(rp, voff[k], voff[k + 1], sms);\n'
                '  return e.bytes();\n}\n')
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + pb.CSRC, src, "-o", so])
    lib = ctypes.CDLL(so)
    lib.estimate.restype = ctypes.c_double
    lib.estimate.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int]

    def run(degrees_of_graphs):
        rp = np.concatenate([[0], np.cumsum(np.concatenate(degrees_of_graphs))]).astype(np.int64)
        voff = np.cumsum([0] + [len(d) for d in degrees_of_graphs]).astype(np.int64)
        return lib.estimate(rp.ctypes.data, voff.ctypes.data, len(degrees_of_graphs), 152)
    return run


def test_chunk_estimate_charges_the_core(estimate):
    below, core = estimate([np.full(30000, 47)]), estimate([np.full(30000, 48)])
    blocks = 2.125 * 30000 * (48 + 127) ** 2
    assert core - below == pytest.approx(2 * 30000 ** 2 + blocks, rel=0.02)
    # the sum of the members' squares, and one chunk of blocks for all
    two = estimate([np.full(30000, 48), np.full(20000, 48)])
    assert two - estimate([np.full(30000, 47), np.full(20000, 47)]) == pytest.approx(
        2 * (30000 ** 2 + 20000 ** 2) + 2.125 * min(2 << 30, 50000 * 175 ** 2), rel=0.02)
    # 32-bit counts; no core beyond the limit of W
    hub = [np.concatenate([np.full(30000, 48), [70000]])]
    assert estimate(hub) > 4 * 30000 ** 2 + 3.125 * blocks / 2.125
    assert estimate([np.full(200000, 48)]) < 2 * 200000 ** 2


ON_THE_GPU = """
import os, sys
sys.path[:0] = [sys.argv[1], os.path.join(sys.argv[1], "tests")]
import torch
torch.cuda.set_device(0)
import graphgen as gg
from gpu_util import gpu_batch
from test_work_space_estimate import _footprint, _regular
from paper_1610_09411_gb300 import escape as esc
g0 = gg.erdos_renyi(100, 0.1, 1)
esc.census(g0.row_ptr, g0.col, n=g0.n)
graphs = {"rings": [_regular(33000, 60), _regular(9000, 50)], "cl": [gg.chung_lu(60000, 2.1, 16, 6000, 3)],
          "dense": [gg.erdos_renyi(1500, 0.3, 4), gg.complete(200)], "rmat": [gg.config_rmat(16, 2)],
          "hubs": [gg.two_hubs()]}[sys.argv[2]]
os.environ["ESC_CORE_MIN_D"] = "1"
free, _ = torch.cuda.mem_get_info()
gpu_batch(graphs)
used = free - torch.cuda.mem_get_info()[0]        # released buffers are kept, each was in use once
need = sum(map(_footprint, graphs))
print(sys.argv[2], "used", used, "estimated", need)
assert used <= need
"""


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["rings", "cl", "dense", "rmat", "hubs"])
def test_what_a_census_takes_stays_below_its_footprint(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", ON_THE_GPU, ROOT, name], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
