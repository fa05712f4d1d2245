"""bench.py's FP64 rooflines divide counts of executed operations, which hold for the captured kernels and call only."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_executed_flops_follow_the_sources_and_the_call(monkeypatch, tmp_path):
    for process, ng in (("ggtt", 0), ("ggttg", 1), ("ggttgg", 2), ("ggttggg", 3)):
        full = 12 if ng == 0 else 1 << (ng + 4)
        assert bench.executed_fp64_flops(process, full, True) > 1000
        assert bench.executed_fp64_flops(process, full - 1, True) is None          # a partial mask
        assert (bench.executed_fp64_flops(process, full, False) is None) == (ng > 0)   # without the shared items
    changed = tmp_path / "kernel.cuh"
    changed.write_text("x")
    monkeypatch.setattr(bench, "ME_SOURCES", (str(changed),))
    assert bench.executed_fp64_flops("ggttg", 32, True) is None                     # other kernel sources


def test_no_achieved_rate_without_executed_counts():
    r = bench.fp64_roofline(None, 311232, 1000, 1.0, 1.25e12, None, "k")
    assert r["achieved"] is None and r["frac"] is None and r["count_ratio"] is None
    r = bench.fp64_roofline(17040.0, 311232, 524288, 9.0, 1.25e12, None, "k")
    assert abs(r["frac"] - 17040 * 524288 / 9.0e-3 / 1.25e12) < 1e-12
