"""The line bench.py prints fits a bounded tail of its output and keeps the headline's figures whole."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

X = 123456789.12345678


def record():
    """A full record of the default run's shape, every number at its longest."""
    part = {"pipe": "fp32", "flops_per_call": X, "peak_tflops": X, "peak_source": "s" * 80}
    roof = {"bound": "alu", "achieved": X, "peak": X, "unit": "TFLOP/s", "frac": X, "traffic": X, "kernel": "k" * 120,
            "flops_per_event": X, "peak_source": "s" * 80, "oracle_flops_per_event": X, "oracle_count_achieved": X,
            "oracle_count_frac": X, "count_ratio": X, "parts": [part] * 3}
    mode = {"value": X, "ms_per_step": X, "me_kernel_ms": X, "value_me_only": X, "steps": 20, "launches_per_step": X,
            "roofline": roof, "rel_err_vs_fp64": {"max": X, "p99": X, "median": X}}
    names = [m for m, _ in bench.MODES]
    leg = {"events_per_gpu": 524288, "seed": 4, "good_helicities": 128, "modes": {m: mode for m in names},
           "launch_shapes": {m: {"flags": 39, "tile_ev": 128} for m in names},
           "epilogues": {"lhe_ms": X, "lhe_MEs_per_s": X, "sde_ms": X, "sde_events_per_s": X, "what": "w" * 200}}
    served = {"slots": 8, "capacity_req_per_s": X, "closed_loop_MEs_per_s": X, "open_loop_rate_req_per_s": X,
              "open_loop_MEs_per_s": X, "p50_ms": X, "p99_ms": X, "peak": {"completed": 1}, "speedup": X}
    clock = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 100, "gpu": "GPU-" + "0" * 36}
    return {"metric": bench.METRIC, "value": X, "unit": "MEs/s", "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": X,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "w" * 110, "process": "ggttg", "events_per_gpu": 524288, "seed": 2, "step": "s" * 90,
                       "l2": "l" * 80, "parallelism": "dp8 (disjoint event ranges)"},
            "me_kernel_ms": X, "wall_s": X, "nonconverged_events": 0, "good_helicities": 32,
            "modes": {m: mode for m in names[1:]}, "launch_shapes": {}, "processes": {p: leg for p in bench.WORKLOADS},
            "serving": {"served_fp64": served, "served_mixed": served, "one_at_a_time_fp64": served, "workload": "w" * 200},
            "graph_batch": {"workload": "w" * 200, "events": 1, "one_launch_sequence_per_job": {"ms": X, "MEs_per_s": X},
                            "graph_branches": {"ms": X, "MEs_per_s": X}, "graph_persistent": {"ms": X, "MEs_per_s": X}},
            "graph": {"ms_per_step": X, "value": X, "same_result": True, "what": "w" * 80},
            "e2e": {"value": X, "unit": "MEs/s", "h2d_bytes_per_step": 83886080, "d2h_bytes_per_step": 4194304, "api": "a" * 100,
                    "mixed": {"value": X, "ms_per_call": X, "device_me_ms": X}},
            "roofline": roof, "cpu_baseline": {"value": X, "unit": "MEs/s", "cores": 16, "kind": "oracle", "sample": "s" * 110},
            "clocks": dict(clock, remeasured_after=clock), "peaks": {"fp64_dfma_tflops": X, "fp32_ffma_tflops": X, "what": "w" * 300},
            "gpu_launches": 300}


def test_line_is_short_and_keeps_the_headline():
    full = record()
    line = bench.summary_line(full)
    text = json.dumps(line)
    assert len(text) <= bench.LINE_BYTES < len(json.dumps(full)) and "\n" not in text
    back = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches"):
        assert back[k] == full[k]
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert back["e2e"][k] == full["e2e"][k]
    assert set(back["processes"]) == {"ggtt", "ggttgg", "ggttggg"}


def test_line_without_the_optional_legs():
    full = dict(record(), graph_batch=None, serving=None, cpu_baseline=None, clocks=None)
    full["processes"] = {"ggttg": full["processes"]["ggttg"]}
    line = bench.summary_line(full)
    assert line["clocks"] is None and line["cpu_baseline"] is None and line["processes"] == {}
