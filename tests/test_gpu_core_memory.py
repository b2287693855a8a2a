"""The dense core only saves time: a census whose core does not fit the
device's free memory is counted by the sweeps alone."""
import os
import subprocess
import sys

import pytest

import graphgen as gg
from gpu_util import assert_same_census, gpu_batch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def core(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    monkeypatch.setenv("ESC_CORE_MIN_D", "1")
    monkeypatch.setenv("ESC_CORE_MIN_DEG", "1")
    monkeypatch.setenv("ESC_CORE_CAP", "1500")
    monkeypatch.setenv("ESC_CORE_CHUNK_MB", "4")
    return monkeypatch


def test_a_core_that_does_not_fit_is_left_out(core):
    """Every limit from the layout's arrays to the packed lists, allocated last."""
    from paper_1610_09411_gb300 import escape as esc
    g = gg.config_rmat(13, 7)
    h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
    try:
        core.setenv("ESC_CORE", "1")
        want = esc.escape_census5(h)
        without = esc.escape_last_kernel_launches(h)
        core.delenv("ESC_CORE")
        assert_same_census(esc.escape_census5(h), want)
        full = esc.escape_last_kernel_launches(h)
        assert full > without
        launches = []
        for mb in (1, 2, 4, 8, 10, 12, 14, 16, 18, 20, 22, 24, 28, 32, 48, 64, 1000):
            core.setenv("ESC_CORE_MAX_MB", str(mb))
            assert_same_census(esc.escape_census5(h), want)
            launches.append(esc.escape_last_kernel_launches(h))
        assert launches == sorted(launches) and launches[0] < full and launches[-1] == full
    finally:
        esc.escape_free(h)


def test_a_batch_without_room_for_its_core(core):
    graphs = [gg.complete(60), gg.erdos_renyi(900, 0.2, 4), gg.barabasi_albert(300, 4, 2)]
    core.setenv("ESC_CORE", "1")
    want = gpu_batch(graphs)
    core.delenv("ESC_CORE")
    core.setenv("ESC_CORE_MAX_MB", "1")
    for got, w in zip(gpu_batch(graphs), want):
        assert_same_census(got, w)


FULL_DEVICE = """
import os, sys
sys.path[:0] = [sys.argv[1], os.path.join(sys.argv[1], "tests")]
import torch
torch.cuda.set_device(0)
import graphgen as gg
from gpu_util import assert_same_census, gpu_census
os.environ["ESC_CORE"] = "1"
g = gg.barabasi_albert(33000, 4, 2)
want = gpu_census(g)
del os.environ["ESC_CORE"]
os.environ.update(ESC_CORE_MIN_D="1", ESC_CORE_MIN_DEG="1", ESC_CORE_CHUNK_MB="64")
free, _ = torch.cuda.mem_get_info()
held = torch.empty(free - (3 << 29), dtype=torch.uint8, device="cuda")   # 1.5 GiB are left; W takes 2
assert_same_census(gpu_census(g), want)
print("counted")
"""


def test_census_on_a_nearly_full_device(core):
    """In a process of its own: the buffers kept from earlier calls would make room."""
    for k in ("ESC_CORE_MIN_D", "ESC_CORE_MIN_DEG", "ESC_CORE_CAP", "ESC_CORE_CHUNK_MB"):
        core.delenv(k)
    r = subprocess.run([sys.executable, "-c", FULL_DEVICE, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "counted" in r.stdout, r.stdout + r.stderr
