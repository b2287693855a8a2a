"""cta_per_sm: what the option sets (host side), and the same counts at every value."""
import ctypes
import os
import re
import subprocess

import pytest

import graphgen as gg
from paper_1610_09411_gb300 import build as pb


@pytest.fixture(scope="module")
def grid(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch")
    src, so = str(d / "l.cpp"), str(d / "l.so")
    with open(src, "w") as f:
        f.write('#include "launch.h"\nextern "C" unsigned grid(int fit, int threads, int cta, int sms, int64_t items) {\n'
                '  return esc::persistent_grid(fit, threads, cta, sms, items);\n}\n')
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + pb.CSRC, src, "-o", so])
    lib = ctypes.CDLL(so)
    lib.grid.argtypes = [ctypes.c_int] * 4 + [ctypes.c_int64]
    return lib.grid


def test_cta_per_sm_limits_the_grid(grid):
    assert grid(3, 512, 0, 152, 10 ** 9) == 3 * 152          # not set: as many as fit
    assert grid(3, 512, 1, 152, 10 ** 9) == 152
    assert grid(3, 512, 8, 152, 10 ** 9) == 3 * 152
    assert grid(24, 64, 2, 152, 10 ** 9) == 16 * 152         # 1,024 threads
    assert grid(6, 256, 1, 152, 10 ** 9) == 2 * 152
    assert grid(1, 1024, 1, 152, 10 ** 9) == 152
    assert grid(3, 512, 2, 152, 7) == 7 and grid(0, 512, 0, 4, 100) == 4


def test_every_cycle_sweep_takes_the_option():
    """Each grid of the 4- and 5-cycle items is computed with the caller's value."""
    with open(os.path.join(pb.CSRC, "census.cu")) as f:
        fills = re.findall(r"fill\(\(const void\*\)(k_cycles[45]_\w+)[^;]*;", f.read())
    with open(os.path.join(pb.CSRC, "census.cu")) as f:
        with_option = re.findall(r"fill\(\(const void\*\)(k_cycles[45]_\w+)[^;]*&grid_i, cta\)\);", f.read())
    assert len(fills) >= 8 and fills == with_option


@pytest.mark.gpu
def test_counts_do_not_depend_on_it():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    torch.cuda.set_device(0)
    from paper_1610_09411_gb300 import escape as esc
    for g in (gg.chung_lu(20000, 2.1, 10, 2000, 8), gg.erdos_renyi(600, 0.2, 3)):
        h = esc.escape_load_csr(g.n, g.row_ptr, g.col)
        try:
            want = esc.escape_census5(h)
            for cta in range(1, 9):
                esc.escape_set_options(h, cta_per_sm=cta)
                assert esc.escape_census5(h) == want
        finally:
            esc.escape_free(h)
