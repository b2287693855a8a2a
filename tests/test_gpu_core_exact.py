"""Large entries of the dense core's contraction and of the counts beside it:
hubs that share tens of thousands of leaves, whose census has a closed form.
The hubs are mutually adjacent and the leaves are not, so a subset of vertices
is a set of hubs and, for every other member, the hubs that it is joined to.
"""
import itertools
import math

import numpy as np
import pytest

import graphgen as gg
import oracle
from gpu_util import assert_same_census, gpu_batch


def _hub_graph(hubs, joined):
    """Hubs 0 .. hubs - 1; leaf k is joined to the hubs in the bits of joined[k]."""
    i, j = np.triu_indices(hubs, 1)
    s, d = [i], [j]
    for h in range(hubs):
        leaves = np.nonzero(joined >> h & 1)[0]
        s.append(np.full(len(leaves), h))
        d.append(hubs + leaves)
    return gg.from_edges(hubs + len(joined), np.concatenate(s), np.concatenate(d), f"hubs{hubs}_{len(joined)}")


def _hub_census(hubs, joined):
    """Its census: every choice of hubs and every multiset of leaf kinds, by class."""
    kinds, counts = np.unique(joined, return_counts=True)
    kinds, counts = [int(x) for x in kinds], [int(x) for x in counts]
    out = {}
    for k in (3, 4, 5):
        pairs = list(itertools.combinations(range(k), 2))
        c = [0] * oracle.NCLS[k]
        for a in range(min(k, hubs) + 1):
            for hs in itertools.combinations(range(hubs), a):
                for leaves in itertools.combinations_with_replacement(range(len(kinds)), k - a):
                    ways = math.prod(math.comb(counts[t], leaves.count(t)) for t in set(leaves))
                    mask = 0
                    for bit, (p, q) in enumerate(pairs):
                        if q < a or (p < a and kinds[leaves[q - a]] >> hs[p] & 1):
                            mask |= 1 << bit
                    c[oracle.classify(k, mask)] += ways
        A = oracle.matrix(k)
        out[f"c{k}"] = c
        out[f"n{k}"] = [sum(x * y for x, y in zip(row, c)) for row in A]
    return out


def _random_joined(hubs, leaves, p, seed):
    rng = np.random.default_rng(seed)
    return sum((rng.random(leaves) < p).astype(np.int64) << h for h in range(hubs))


def test_closed_form_equals_the_oracle():
    for hubs, joined in [(3, _random_joined(3, 40, 0.7, 1)), (4, np.full(25, 15)), (2, np.arange(30) % 4)]:
        assert_same_census(_hub_census(hubs, joined), oracle.census(_hub_graph(hubs, joined)))


@pytest.fixture
def core(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)

    def use(min_deg, cap):
        monkeypatch.setenv("ESC_CORE_MIN_D", "1")
        monkeypatch.setenv("ESC_CORE_MIN_DEG", str(min_deg))
        monkeypatch.setenv("ESC_CORE_CAP", str(cap))
    use.env = monkeypatch
    return use


def _census(g, core):
    """The census, and how many more kernels it launched than one without a core."""
    from paper_1610_09411_gb300 import escape as esc
    h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
    try:
        got = esc.escape_census5(h)
        used = esc.escape_last_kernel_launches(h)
        core.env.setenv("ESC_CORE", "1")
        esc.escape_census5(h)
        return got, used - esc.escape_last_kernel_launches(h)
    finally:
        esc.escape_free(h)


@pytest.mark.gpu
@pytest.mark.parametrize("hubs,p", [(4, 0.9), (3, 0.995), (5, 0.5)])
def test_odd_entries_near_the_largest_core(hubs, p, core):
    """Every vertex in the core: sums of up to 2^15 that grow by odd steps."""
    joined = _random_joined(hubs, 32768 - hubs, p, 7 + hubs)
    core(1, 32768)
    got, more = _census(_hub_graph(hubs, joined), core)
    assert more > 0
    assert_same_census(got, _hub_census(hubs, joined))


@pytest.mark.gpu
@pytest.mark.parametrize("hubs,cap", [(4, 4), (3, 3), (5, 4), (4, 200)])
def test_below_core_counts_above_16_bits(hubs, cap, core):
    """Core hubs that share more than 2^16 neighbours below the core."""
    joined = np.full(65600, (1 << hubs) - 1)
    joined[:37] = 1
    core(1, cap)
    got, more = _census(_hub_graph(hubs, joined), core)
    assert more > 0
    assert_same_census(got, _hub_census(hubs, joined))


@pytest.mark.gpu
def test_odd_entries_above_2_to_the_16_in_a_union(core):
    """The core of a union has no vertex limit of its own."""
    joined = [_random_joined(3, 66500, 0.99, 11), _random_joined(4, 300, 0.8, 12)]
    core(1, 32768)
    for j, hubs, got in zip(joined, (3, 4), gpu_batch([_hub_graph(3, joined[0]), _hub_graph(4, joined[1])])):
        assert_same_census(got, _hub_census(hubs, j))
