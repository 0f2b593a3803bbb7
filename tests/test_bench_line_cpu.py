"""bench.py's one line: the measurement alone, short enough that the last 1,500
characters of the output hold all of it, however much is measured beside it; the
rest goes to stderr, a line per part."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _record():
    num = 1234567890.1234567
    big = {f"entry_{i}": {"value": num, "how": "x" * 80} for i in range(40)}
    return {"metric": "PNE terms contracted/sec", "value": num, "unit": "terms/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.58467840254306, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": {"workload": bench.WORKLOADS["random16"]["desc"], "networks_per_step_per_gpu": 32,
                       "terms_per_network": 27216, "clusters_per_network": 9999, "K": 8,
                       "bp_arithmetic": "float-float pairs of FP32 (~2^-48 per operation), FP64 storage",
                       "contraction_dtype": "f64", "term_sums": "FP64",
                       "l2": "flushed between timed steps (256 MB write)",
                       "enumeration": "recomputed every step (cache off)",
                       "parallelism": "independent networks per GPU x1"},
            "e2e": {"value": num, "unit": "terms/s", "h2d_bytes_per_step": 13950744, "d2h_bytes_per_step": 5824,
                    "ms_per_step": 0.6194815993309021},
            "gpu_launches": 480, "host_ms_per_step": big, "roofline": {"kernel": "bp_sweeps", "bound": "alu",
                                                                     "frac": 0.1066308, **big},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 2}, "variants": big,
            "peaks_measured": big, "cpu_baseline": {"value": num, "unit": "terms/s", "cores": 16, "kind": "oracle",
                                                    "sample": "y" * 400, "single_thread": big},
            "workloads": {"one": big, "two": big}}


def test_the_line_is_whole_and_short(capsys, tmp_path):
    out = _record()
    bench.emit(out, str(tmp_path / "all.json"))
    cap = capsys.readouterr()
    lines = cap.out.splitlines()
    assert len(lines) == 1 and len(lines[0]) <= 1500
    d = json.loads(lines[0])
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "e2e", "gpu_launches", "clocks"):
        assert d[k] == out[k]
    assert d["config"]["workload"] == out["config"]["workload"] and d["config"]["l2"] == out["config"]["l2"]
    told = {}
    for ln in cap.err.splitlines():
        told.update(json.loads(ln))
    for k in ("host_ms_per_step", "roofline", "variants", "peaks_measured", "cpu_baseline", "config"):
        assert told[k] == out[k]
    assert told["one"] == out["workloads"]["one"] and told["two"] == out["workloads"]["two"]
    assert json.load(open(tmp_path / "all.json")) == out
