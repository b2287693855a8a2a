"""The dense core of the pair and wheel sweeps (operand blocks, tensor-core
contraction, the split between it and the sweeps) against the oracle and
against the sweeps alone, at the sizes where tiles, blocks, chunks and the
core's edge can go wrong.  Counts are whole numbers: every comparison is exact.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle
from gpu_util import assert_same_census, gpu_census

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    from paper_1610_09411_gb300 import build
    build.build()


def _core(monkeypatch, min_deg, cap, chunk_mb=2048):
    monkeypatch.setenv("ESC_CORE_MIN_D", "1")
    monkeypatch.setenv("ESC_CORE_MIN_DEG", str(min_deg))
    monkeypatch.setenv("ESC_CORE_CAP", str(cap))
    monkeypatch.setenv("ESC_CORE_CHUNK_MB", str(chunk_mb))


GRAPHS = {
    "er": lambda: gg.erdos_renyi(300, 0.3, 5),
    "cl": lambda: gg.chung_lu(3000, 2.1, 12, 700, 3),
    "K150": lambda: gg.complete(150),
    "bipartite": lambda: gg.complete_bipartite(40, 90),
    "rmat": lambda: gg.config_rmat(10, 3),
}
_oracle = {}


@pytest.mark.parametrize("min_deg,cap", [(1, 100000), (2, 130), (1, 127), (1, 129), (40, 257), (1, 1), (1, 3)])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_core_edges_match_the_oracle(name, min_deg, cap, monkeypatch):
    """Cores of every size from one vertex to the whole graph, around the
    128-row and 256-column tile edges."""
    _core(monkeypatch, min_deg, cap)
    g = GRAPHS[name]()
    if name not in _oracle:
        _oracle[name] = oracle.census(g)
    assert_same_census(gpu_census(g), _oracle[name])


@pytest.mark.parametrize("cap,chunk_mb,warp_max", [(1500, 1, 64), (400, 2048, 1), (3000, 1, 1024)])
def test_core_chunks_and_wheel_groups_match_the_sweeps_alone(cap, chunk_mb, warp_max, monkeypatch):
    """Several chunks of operand blocks, centres counted by warps and by groups
    of one or more warps of a CTA, against the census without a core."""
    g = gg.config_rmat(13, 7)
    monkeypatch.setenv("ESC_CORE", "1")
    want = gpu_census(g)
    monkeypatch.delenv("ESC_CORE")
    monkeypatch.setenv("ESC_WHEEL_WARP_MAX", str(warp_max))
    _core(monkeypatch, 2, cap, chunk_mb)
    assert_same_census(gpu_census(g), want)


@pytest.mark.parametrize("mode", ["3", "2", "1"])
def test_core_with_counts_above_16_bits(mode, monkeypatch):
    """Degrees of 2^16 and more: 32-bit wedge counts and below-core counts."""
    monkeypatch.setenv("ESC_PAIR_WINDOW", mode)
    g = gg.two_hubs()
    monkeypatch.setenv("ESC_CORE", "1")
    want = gpu_census(g)
    monkeypatch.delenv("ESC_CORE")
    for cap in (2, 30, 600):
        _core(monkeypatch, 1, cap)
        assert_same_census(gpu_census(g), want)


@pytest.mark.parametrize("mode", ["3", "2", "1"])
@pytest.mark.parametrize("min_deg", [1, 20])
def test_core_of_a_batch_matches_the_oracle(min_deg, mode, monkeypatch):
    """One square of wedge counts per member, members with and without core vertices."""
    from paper_1610_09411_gb300 import escape as esc
    monkeypatch.setenv("ESC_PAIR_WINDOW", mode)
    _core(monkeypatch, min_deg, 100000, 1)
    graphs = [gg.complete(40), gg.erdos_renyi(150, 0.4, 4), gg.empty(2), gg.barabasi_albert(120, 4, 2),
              gg.chung_lu(400, 2.1, 8, 80, 6), gg.petersen(), gg.complete(140)]
    voff = np.cumsum([0] + [g.n for g in graphs]).astype(np.int64)
    base = np.cumsum([0] + [g.nnz for g in graphs])
    rp = np.concatenate([g.row_ptr[:-1] + b for g, b in zip(graphs, base)] + [base[-1:]]).astype(np.int64)
    col = np.concatenate([g.col for g in graphs]).astype(np.int32)
    for g, r in zip(graphs, esc.escape_census5_batch(voff, rp, col)):
        assert_same_census(r, oracle.census(g))
