"""The benchmark's figures from profiler summaries count only for the kernel source that
was profiled."""
import hashlib
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
bench = pytest.importorskip("bench")


def test_profiled_figures_belong_to_the_kernel_source(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2108_12742_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    (csrc / "sweep.cuh").write_text("kernel")
    sha = hashlib.sha256(b"kernel").hexdigest()
    (tmp_path / "profiles" / "s.md").write_text(
        "| warp instructions x 32 per cell | 1060 |\n"
        "| FP64-unit warp instructions x 32 per cell | 143.2 |\n"
        f"traffic_bytes_per_launch_4096: 1.5e9\nsource_sha256: {sha}\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profiled("s.md", bench.INST) == 1060
    assert bench.profiled("s.md", bench.FP64_INST) == 143.2
    assert bench.profiled("s.md", bench.TRAFFIC) == 1.5e9
    assert bench.profiled("none.md", bench.INST) is None
    (csrc / "sweep.cuh").write_text("another kernel")
    for pattern in (bench.INST, bench.FP64_INST, bench.TRAFFIC):
        assert bench.profiled("s.md", pattern) is None


def test_fp64_roofline_needs_a_count_of_the_present_kernel():
    r = bench.fp64_roofline(2.0, 1000000, 1.26, None)
    assert r["frac"] is None and r["achieved"] is None and r["kernel_ms"] == 2.0
    r = bench.fp64_roofline(2.0, 1000000, 1.26, 143.0)
    assert r["achieved"] == pytest.approx(0.143) and r["frac"] == pytest.approx(0.143 / 1.26)
