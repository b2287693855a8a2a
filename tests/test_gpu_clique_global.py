"""Out-degrees whose bit matrix does not fit shared memory: counts of complete
multipartite graphs, and the rate of the 5-clique loop."""
import itertools
import math

import numpy as np
import pytest

import graphgen as gg
import oracle
from gpu_util import assert_same_census, gpu_census


def _multipartite(parts, size):
    i, j = np.triu_indices(parts * size, 1)
    keep = i % parts != j % parts               # members of a part are spread over the ids
    return gg.from_edges(parts * size, i[keep], j[keep], f"multipartite{parts}x{size}")


def _multipartite_census(parts, size):
    """Closed form: a k-subset is a way to split k over the parts."""
    out = {}
    for k in (3, 4, 5):
        c = [0] * oracle.NCLS[k]
        pairs = list(itertools.combinations(range(k), 2))
        for split in _partitions(k, k):
            if max(split) > size or len(split) > parts:
                continue
            ways = math.comb(parts, len(split)) * math.factorial(len(split))
            for x in set(split):
                ways //= math.factorial(split.count(x))
            for x in split:
                ways *= math.comb(size, x)
            part = [t for t, x in enumerate(split) for _ in range(x)]
            c[oracle.classify(k, sum(1 << b for b, (p, q) in enumerate(pairs) if part[p] != part[q]))] += ways
        A = oracle.matrix(k)
        out[f"c{k}"], out[f"n{k}"] = c, [sum(x * y for x, y in zip(row, c)) for row in A]
    return out


def _partitions(n, most):
    if n == 0:
        return [[]]
    return [[x] + rest for x in range(min(n, most), 0, -1) for rest in _partitions(n - x, x)]


@pytest.fixture
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)


def test_closed_form_equals_the_oracle():
    for parts, size in [(4, 3), (9, 2), (3, 7), (12, 1)]:
        assert_same_census(_multipartite_census(parts, size), oracle.census(_multipartite(parts, size)))


# out-degrees of up to 1,377, 1,398 and 1,200: the last words of a row partly used, full and nearly empty
@pytest.mark.gpu
@pytest.mark.parametrize("parts,size", [(460, 3), (700, 2), (13, 100)])
@pytest.mark.parametrize("core", ["1", "2"])
def test_multipartite_beyond_the_shared_memory_bit_matrix(parts, size, core, gpu, monkeypatch):
    monkeypatch.setenv("ESC_CORE", core)
    assert_same_census(gpu_census(_multipartite(parts, size)), _multipartite_census(parts, size))


@pytest.mark.gpu
def test_rate_beyond_the_shared_memory_bit_matrix(gpu):
    """The 5-clique loop's work on K_n grows with n^4 words of n / 64: on a matrix
    in global memory it takes no longer per word than on one in shared memory."""
    from paper_1610_09411_gb300 import escape as esc
    ms = {}
    for n in (1000, 1500):
        g = gg.complete(n)
        h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
        try:
            esc.escape_set_options(h, serial_phases=True)
            for _ in range(2):
                esc.escape_census5(h)
                ms[n] = min(ms.get(n, 1e9), esc.escape_last_phase_ms(h)["cliques"])
        finally:
            esc.escape_free(h)
    assert ms[1500] <= 1.5 ** 5 * ms[1000], ms
