"""bench.py's rates of work: the byte model is the method's, not what the
kernels read, so it is no fraction of a bandwidth; the traffic record of the
pair phase follows core.cu too."""
import os
import shutil

import pytest

import bench
import graphgen as gg


def test_rates_of_work_are_no_bandwidth(monkeypatch):
    sums = {"W": 10 ** 9, "D": 12 * 10 ** 9, "T": 10 ** 8}
    phases = {"pairs": 50.0, "wheels": 20.0, "cliques": 30.0, "cycles5": 40.0}
    roof = bench.dominant_phase("rmat22", sums, phases, {"pairs": 25.0})
    assert roof["kernel"] == "k_pairs" and roof["frac"] is None and "model" in roof["unit"]
    assert roof["achieved"] == pytest.approx(4 * 13.0 / 0.05) and roof["achieved_alone"] == pytest.approx(4 * 13.0 / 0.025)
    assert bench.dominant_phase("rmat22", None, phases, {}) is None
    monkeypatch.setattr(bench, "stored_traffic", lambda kernel, workload: 5 * 10 ** 9)
    monkeypatch.setattr(bench, "measured_peak", lambda: (1000.0, "measured"))
    roof = bench.dominant_phase("rmat22", sums, phases, {"pairs": 25.0})
    assert roof["traffic_gbs"] == pytest.approx(200.0) and roof["traffic_frac"] == pytest.approx(0.2)
    g = gg.erdos_renyi(200, 0.1, 1)
    work = bench.census_work(g, {"W": 5, "D": 7}, 2.0)
    total, terms = bench.census_alg_bytes(g, {"W": 5, "D": 7})
    assert work["frac"] is None and work["achieved"] == pytest.approx(total / 2e-3 / 1e9)
    assert bench.census_work(g, None, 2.0) is None


def test_digest_of_the_pair_phase_covers_the_core(tmp_path, monkeypatch):
    src = os.path.join(bench.ROOT, "paper_1610_09411_gb300", "csrc")
    dst = tmp_path / "paper_1610_09411_gb300" / "csrc"
    dst.mkdir(parents=True)
    for name in ("census.cu", "core.cu"):
        shutil.copy(os.path.join(src, name), dst / name)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    base = bench.source_digest("k_pairs")
    with open(dst / "core.cu", "a") as f:
        f.write("// changed\n")
    assert bench.source_digest("k_pairs") != base
