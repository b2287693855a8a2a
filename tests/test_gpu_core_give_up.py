"""A wait of the dense core's contraction that runs out: the call ends with
ETIMEOUT once what is in flight has landed, and the next one counts as usual.
The reading warps take one of their waits as run out, with operand copies and
MMAs of the tiles behind it under way; the other roles then wait for what does
not come, up to a short limit."""
import pytest

import graphgen as gg
from gpu_util import assert_same_census, gpu_batch, gpu_census

pytestmark = pytest.mark.gpu

ETIMEOUT = 5


@pytest.fixture
def core(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    monkeypatch.setenv("ESC_CORE_MIN_D", "1")
    monkeypatch.setenv("ESC_CORE_MIN_DEG", "1")
    return monkeypatch


# K700: three row blocks by two of columns per centre; the R-MAT core leaves vertices below it, in several chunks
@pytest.mark.parametrize("name,cap,chunk_mb,give_up", [("K700", 100000, 2048, 1), ("K700", 100000, 2048, 2),
                                                       ("K700", 100000, 2048, 9), ("rmat", 600, 1, 1),
                                                       ("rmat", 600, 2048, 1), ("rmat", 600, 2048, 3)])
def test_a_wait_that_runs_out_gives_a_timeout(name, cap, chunk_mb, give_up, core):
    from paper_1610_09411_gb300.escape import EscapeError
    g = gg.complete(700) if name == "K700" else gg.config_rmat(13, 7)
    core.setenv("ESC_CORE_CAP", str(cap))
    core.setenv("ESC_CORE_CHUNK_MB", str(chunk_mb))
    want = gpu_census(g)
    core.setenv("ESC_CORE_WAIT_US", "2000")
    core.setenv("ESC_CORE_GIVE_UP", str(give_up))
    with pytest.raises(EscapeError) as e:
        gpu_census(g)
    assert e.value.code == ETIMEOUT
    core.delenv("ESC_CORE_WAIT_US")
    core.delenv("ESC_CORE_GIVE_UP")
    assert_same_census(gpu_census(g), want)


def test_a_batch_reports_it_too(core):
    from paper_1610_09411_gb300.escape import EscapeError
    graphs = [gg.complete(300), gg.erdos_renyi(200, 0.3, 4)]
    core.setenv("ESC_CORE_WAIT_US", "2000")
    core.setenv("ESC_CORE_GIVE_UP", "1")
    with pytest.raises(EscapeError) as e:
        gpu_batch(graphs)
    assert e.value.code == ETIMEOUT
