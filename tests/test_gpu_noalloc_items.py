"""escape_cycles4_noalloc at the edges of its item classes (rows of 31, 32 and
33 entries, one and no entries, the largest graph) and with malformed ids and
offsets, which must be reported and never followed.  Counts are exact."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    from paper_1610_09411_gb300 import build
    build.build()


def _run(n, row_ptr, col):
    import torch
    from paper_1610_09411_gb300 import escape as esc
    rp, c = torch.from_numpy(row_ptr).cuda(), torch.from_numpy(col).cuda()
    v = torch.full((max(n, 1),), 5, dtype=torch.int64, device="cuda")
    t = torch.full((1,), 5, dtype=torch.int64, device="cuda")
    esc.escape_cycles4_noalloc(n, rp, c, v, t)
    return v.cpu().numpy()[:n].astype(np.uint64), int(t.item())


@pytest.mark.parametrize("make", [
    lambda: gg.complete(32), lambda: gg.complete(33), lambda: gg.complete(34),
    lambda: gg.complete_bipartite(32, 33), lambda: gg.complete_bipartite(2, 300), lambda: gg.star(40),
    lambda: gg.cycle(4), lambda: gg.path(3), lambda: gg.empty(9), lambda: gg.chung_lu(9001, 2.1, 14, 3000, 5),
], ids=["K32", "K33", "K34", "K32,33", "K2,300", "star", "C4", "P3", "empty", "cl"])
def test_noalloc_item_classes_match_the_oracle(make):
    g = make()
    want = oracle.census(g, per_element=True)
    v, total = _run(g.n, g.row_ptr, g.col if g.col.size else np.zeros(1, np.int32))
    assert np.array_equal(v, np.asarray(want["per_element"]["C4_i"], dtype=np.uint64))
    assert total == want["n4"][3]


@pytest.mark.parametrize("break_it", ["id_high", "id_negative", "single_row_id", "offset_high", "offset_decreasing"])
def test_noalloc_reports_malformed_rows(break_it):
    """The kernels' own checks skip the access and the call returns EINVAL."""
    from paper_1610_09411_gb300 import escape as esc
    g = gg.complete(40) if break_it != "single_row_id" else gg.path(2)
    rp, col = g.row_ptr.copy(), g.col.copy()
    if break_it == "id_high":
        col[7] = g.n
    elif break_it == "id_negative":
        col[7] = -1
    elif break_it == "single_row_id":
        col[0] = 12
    elif break_it == "offset_high":
        rp[3] = rp[-1] + 5
    else:
        rp[3] = rp[2] - 1
    with pytest.raises(esc.EscapeError) as ei:
        _run(g.n, rp, col)
    assert ei.value.code == 1
