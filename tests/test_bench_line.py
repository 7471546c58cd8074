"""The line that the benchmark prints: the headline's keys, parseable, and short
enough to be whole in the last 3,000 characters of the output."""
import json

import bench


def _result(long):
    text = "x" * long
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 41}
    bed = {"ms_per_step": 0.4737283, "value": 1.0, "stages_ms": {text: 1.0}}
    return {"metric": bench.METRIC, "value": 211091234.56789, "unit": "particle updates/s",
            "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 0.47372831234,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64",
            "data": "synthetic", "config": {"workload": bench.WORKLOAD, "mesh": text[:200]},
            "run": {"precision": "mixed", "launch": text}, "gpu_launches": 760,
            "gpu_launches_note": text, "clocks": clocks, "mixed": bed, "fp64": bed,
            "e2e": {"value": 1.5e8, "unit": "particle updates/s", "h2d_bytes_per_step": 32783648,
                    "d2h_bytes_per_step": 5545728, "clocks": clocks},
            "err_mixed_vs_fp64": {"eps_h": 1e-7, "f": 2e-7},
            "cpu_baseline": {"value": 89861.9, "sample": text},
            "roofline": {"bound": "alu", "frac": 0.046, "kernel": "k", "others": {text: text}},
            "workloads": {"q3_24x24x96_1m": {"mixed": bed, "roofline": {text: 1.0}},
                          "dem": {"ms_per_step": 0.77, "status": text}}}


def test_line_is_short_and_has_the_headline():
    for long in (10, 1000, 20000):
        res = _result(long)
        line = bench.headline(res)
        assert "\n" not in line and len(line) <= 2800
        d = json.loads(line)
        for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
                  "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config",
                  "gpu_launches", "clocks", "e2e"):
            assert d[k] == res[k]
    assert json.loads(bench.headline(_result(10)))["workloads_ms_per_step"] == {
        "q3_24x24x96_1m": 0.4737283, "dem": 0.77}
