"""The benchmark's result line stays short however many settings its sweep tries."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_result_line_is_short_and_keeps_the_figures():
    import bench

    x = 0.4320000112056732
    point = {"ef": 64, "tau": 0.9, "recall": 0.985, "ms": x, "mean_expansions": 37.035400390625,
             "entry": True, "stop": {"stop_min": 8, "stop_every": 4}}
    stats = {"min": x, "median": x, "max": x}
    note = "first 40 of the 10,000 queries, exact fused top-10 over all 1,000,000 objects " * 2
    kept = {"metric": "QPS at Recall@10 >= 0.95 (hybrid recall, Sec. 6.1) on 1 GB300",
            "value": 22262345.123456789, "unit": "queries/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": x, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {f"key_{i}": note[:60] for i in range(14)},
            "roofline": {"bound": "hbm", "unit": "GB/s", "step_ms": stats,
                         **{f"figure_{i}": x for i in range(9)}},
            "e2e": {"value": 19586827.623393696, "unit": "queries/s",
                    "h2d_bytes_per_step": 5150000, "d2h_bytes_per_step": 900000, "recall": x},
            "gpu_launches": 60, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0,
                                           "power_w_max": 206.22, "samples": 3, "reasons": []}}
    line = dict(kept, sweep=[point] * 200, learned={"sweep": [point] * 200},
                plain_f32={"qps": x},
                brute_force={"bound": "alu", "ms": x, "achieved": x, "peak": x,
                             "unit": "TFLOP/s", "frac": x, "peak_kind": note},
                cpu_baseline={"value": x, "unit": "queries/s", "cores": 1, "kind": "oracle",
                              "sample": note, "all_cores": {"value": x, "sample": note},
                              "search": {"value": x, "sample": note}})
    short, details = bench.split_details(line)
    assert len(json.dumps(short)) < 2500
    for key, value in kept.items():
        if isinstance(value, float):
            assert abs(short[key] / value - 1) < 1e-6
        elif not isinstance(value, dict):
            assert short[key] == value
    assert set(short["e2e"]) == set(kept["e2e"]) and set(short["clocks"]) == set(kept["clocks"])
    assert short["cpu_baseline"]["search"] == short["brute_force"]["ms"] == short["ms_per_step"]
    assert details["sweep"] == line["sweep"] and details["cpu_baseline"] == line["cpu_baseline"]
