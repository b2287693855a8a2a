"""Medium items of small graphs counted by place in the graph, against the
hash tables (ESC_DIRECT=1) and the oracle: single graphs at the size limit, one
vertex above it, and unions with empty and edgeless members.  Exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from gpu_util import assert_same_census, gpu_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    from paper_1610_09411_gb300 import build
    build.build()


def _no_light(monkeypatch):
    for sweep in ("PAIR", "CYCLE"):
        monkeypatch.setenv(f"ESC_{sweep}_SMALL_W", "1")


GRAPHS = {
    "K70": lambda: gg.complete(70),
    "bipartite": lambda: gg.complete_bipartite(33, 64),
    "star": lambda: gg.star(1100),
    "er": lambda: gg.erdos_renyi(261, 0.2, 5),
    "cl8191": lambda: gg.chung_lu(8191, 2.2, 8, 1500, 3),
    "cl8192": lambda: gg.chung_lu(8192, 2.2, 8, 1500, 4),
    "cl8193": lambda: gg.chung_lu(8193, 2.2, 8, 1500, 5),
}


@pytest.mark.parametrize("hash_only", [False, True], ids=["direct", "hash"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_direct_items_match_the_oracle(name, hash_only, monkeypatch):
    from paper_1610_09411_gb300 import escape as esc
    _no_light(monkeypatch)
    if hash_only:
        monkeypatch.setenv("ESC_DIRECT", "1")
    g = GRAPHS[name]()
    want = oracle.census(g, per_element=True)
    got = esc.census(g.row_ptr, g.col, n=g.n, per_element=True)
    assert_same_census(got, want)
    for k in ("C4_e", "C4_i", "K4_e"):
        assert np.array_equal(got["per_element"][k], np.asarray(want["per_element"][k], dtype=np.uint64)), k


@pytest.mark.parametrize("core", [False, True])
@pytest.mark.parametrize("hash_only", [False, True], ids=["direct", "hash"])
def test_direct_union_matches_the_oracle(hash_only, core, monkeypatch):
    _no_light(monkeypatch)
    if hash_only:
        monkeypatch.setenv("ESC_DIRECT", "1")
    if core:
        monkeypatch.setenv("ESC_CORE_MIN_D", "1")
        monkeypatch.setenv("ESC_CORE_MIN_DEG", "20")
    graphs = [gg.complete(30), gg.empty(0), gg.erdos_renyi(150, 0.3, 4), gg.empty(2), gg.barabasi_albert(120, 4, 2),
              gg.star(90), gg.chung_lu(400, 2.1, 8, 80, 6), gg.complete(3), gg.erdos_renyi(333, 0.15, 7)]
    for g, r in zip(graphs, gpu_batch(graphs)):
        assert_same_census(r, oracle.census(g))


def test_sparse_union_with_more_graphs_than_edges():
    """Too sparse for the sort by graph: the general path."""
    graphs = [gg.empty(1)] * 40 + [gg.path(4), gg.cycle(5), gg.empty(0), gg.complete(4)]
    for g, r in zip(graphs, gpu_batch(graphs)):
        assert_same_census(r, oracle.census(g))


@pytest.mark.parametrize("words", [4000, None], ids=["large_hash", "one_window"])
def test_large_pair_items_match_the_oracle(words, monkeypatch):
    """Pair items of 8,193 to 24,576 counters: hashed when a window does not
    hold the graph's ranks."""
    from paper_1610_09411_gb300 import escape as esc
    if words:
        monkeypatch.setenv("ESC_PAIR_WIN_WORDS", str(words))
    g = gg.chung_lu(26001, 2.1, 12, 3000, 9)
    assert_same_census(esc.census(g.row_ptr, g.col, n=g.n), oracle.census(g))
