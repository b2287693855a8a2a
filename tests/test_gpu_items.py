"""Item classes of the pair, 4-cycle and 5-cycle sweeps (packed hash tables for
light and medium items, shared-memory windows for heavy ones) against the
oracle, per-element arrays included.  Counts are whole numbers: exact."""
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


GRAPHS = {
    "er": lambda: gg.erdos_renyi(260, 0.2, 5),
    "cl": lambda: gg.chung_lu(4000, 2.1, 12, 700, 3),
    "star": lambda: gg.star(1100),
    "bipartite": lambda: gg.complete_bipartite(33, 64),
    "K70": lambda: gg.complete(70),
    "n127": lambda: gg.erdos_renyi(127, 0.5, 2),       # n + 1 a power of two: the widest rank of a packed word
    "n128": lambda: gg.erdos_renyi(128, 0.5, 3),
}
_oracle = {}


def _check(name):
    from paper_1610_09411_gb300 import escape as esc
    g = GRAPHS[name]()
    if name not in _oracle:
        _oracle[name] = oracle.census(g, per_element=True)
    want = _oracle[name]
    got = esc.census(g.row_ptr, g.col, n=g.n, per_element=True)
    assert_same_census(got, want)
    for k in ("T_e", "C4_e", "K4_e", "t_i", "C4_i", "K4_i"):
        assert np.array_equal(got["per_element"][k], np.asarray(want["per_element"][k], dtype=np.uint64)), k


@pytest.mark.parametrize("small,large", [(1, 1), (1, 65), (33, 33), (65, 100000), (100000, 100000)])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_item_classes_match_the_oracle(name, small, large, monkeypatch):
    """Every class on every graph: limits 0 (all heavy) up to the tables' sizes."""
    for sweep in ("PAIR", "CYCLE"):
        monkeypatch.setenv(f"ESC_{sweep}_SMALL_W", str(small))
        monkeypatch.setenv(f"ESC_{sweep}_LARGE_W", str(large))
    _check(name)


@pytest.mark.parametrize("words", [4, 60, 500])
@pytest.mark.parametrize("name", ["er", "cl", "bipartite"])
def test_heavy_cycle_items_in_narrow_windows(name, words, monkeypatch):
    for sweep in ("PAIR", "CYCLE"):
        monkeypatch.setenv(f"ESC_{sweep}_SMALL_W", "1")
        monkeypatch.setenv(f"ESC_{sweep}_LARGE_W", "1")
        monkeypatch.setenv(f"ESC_{sweep}_WIN_WORDS", str(words))
    _check(name)


def test_two_hubs_heavy_cycles(monkeypatch):
    """Counts above 2^16: the 64-bit counters beside the windows."""
    g = gg.two_hubs()
    want = gpu_census(g)
    for sweep in ("PAIR", "CYCLE"):
        monkeypatch.setenv(f"ESC_{sweep}_SMALL_W", "1")
        monkeypatch.setenv(f"ESC_{sweep}_LARGE_W", "1")
        monkeypatch.setenv(f"ESC_{sweep}_WIN_WORDS", "400")
    assert_same_census(gpu_census(g), want)


@pytest.mark.parametrize("limit", ["1", "40", "100000"])
def test_batch_item_classes_match_the_oracle(limit, monkeypatch):
    from paper_1610_09411_gb300 import escape as esc
    for sweep in ("PAIR", "CYCLE"):
        monkeypatch.setenv(f"ESC_{sweep}_SMALL_W", limit)
        monkeypatch.setenv(f"ESC_{sweep}_LARGE_W", limit)
    graphs = [gg.complete(30), gg.erdos_renyi(150, 0.3, 4), gg.empty(2), gg.barabasi_albert(120, 4, 2), gg.star(90),
              gg.chung_lu(400, 2.1, 8, 80, 6), gg.petersen(), gg.cycle(5)]
    voff = np.cumsum([0] + [g.n for g in graphs]).astype(np.int64)
    base = np.cumsum([0] + [g.nnz for g in graphs])
    rp = np.concatenate([g.row_ptr[:-1] + b for g, b in zip(graphs, base)] + [base[-1:]]).astype(np.int64)
    col = np.concatenate([g.col for g in graphs]).astype(np.int32)
    for g, r in zip(graphs, esc.escape_census5_batch(voff, rp, col)):
        assert_same_census(r, oracle.census(g))
