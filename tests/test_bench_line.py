"""The benchmark's line on stdout stays short enough for a reader that keeps a few
kilobytes, however long the studies are, and holds the measurement whole."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def result():
    text = "x" * 120
    res = {"metric": bench.HEADLINE_METRIC, "value": 1.3e10, "unit": "walk steps/s", "n_gpus": 1, "steps": 20, "warmup": 5,
           "ms_per_step": 3015.2390136, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "u64 counts, f64 finalize", "data": "synthetic",
           "config": {"workload": text, "n": 10 ** 6, "arcs": 10 ** 7, "kernel": text, "l2": text, "parallelism": text},
           "walk_steps": {"wilson": 10 ** 11, "uniform_walk": 10 ** 8, "pi_walk": 10 ** 8},
           "roofline": {"bound": "hbm", "achieved": 2.9e3, "traffic_note": text, "kernel": text, "peak_kind": text},
           "gpu_launches": 180, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
           "e2e": {"value": 1.3e10, "unit": "walk steps/s", "h2d_bytes_per_step": 44000004, "d2h_bytes_per_step": 8000008,
                   "note": text},
           "cpu_baseline": {"value": 1.3e8, "unit": "walk steps/s", "cores": 16, "kind": "oracle", "sample": text},
           "time_to_accuracy": {"omega": 4096, "gpu_seconds": 0.0154321, "curve": [{"omega": k} for k in range(400)]},
           "time_to_accuracy_large": [{"workload": "g%d" % k, "plain": {"omega": 1024, "gpu_seconds": 1.5}, "cv": {
               "omega_extrapolated": 5000}} for k in range(100)],
           "spantree": {"trees": 4096, "seconds": 1.7, "trees_per_s": 2400.0, "time_to_accuracy": {"omega": 300000,
                                                                                                 "gpu_seconds": 0.3}},
           "batched": {"seconds": 33.0, "runs": [{"x": text}] * 200}}
    return res


def test_line_is_short_and_whole():
    res = result()
    assert len(json.dumps(res)) > 30000
    line = bench.stdout_line(res)
    assert "\n" not in line and len(line) <= bench.LINE_BYTES
    d = json.loads(line)
    for k in bench.LINE_KEYS:
        assert (k in d) == (k in res) and d.get(k) == res.get(k)
    assert d["studies"]["time_to_accuracy"] == {"omega": 4096, "gpu_seconds": 0.01543}
