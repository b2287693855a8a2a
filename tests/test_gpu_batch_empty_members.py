"""A batch of one dense graph among very many empty ones: the core's layout has
no room for the graphs, the census has."""
import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle
from gpu_util import assert_same_census

pytestmark = pytest.mark.gpu


# 10 members, and more than 4 MiB of 64-bit words
@pytest.mark.parametrize("empty", [9, 600000])
def test_dense_graph_among_empty_ones(empty):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    from paper_1610_09411_gb300 import escape as esc
    g = gg.complete(120)                         # 4.9e7 diamonds: above the core's limits
    voff = np.full(empty + 2, g.n, dtype=np.int64)
    voff[0] = 0
    rp, col = g.row_ptr.astype(np.int64), g.col.astype(np.int32)
    out = (esc.Census * (empty + 1))()
    code = esc.LIB.escape_census5_batch(empty + 1, voff.ctypes.data, rp.ctypes.data, col.ctypes.data, 0, out, None)
    assert code == 0
    assert_same_census(out[0].to_dict(), oracle.census(g))
    words = np.frombuffer(out, dtype=np.uint64)[ctypes.sizeof(esc.Census) // 8:]
    assert not words.any()                       # no subsets in a graph without vertices
