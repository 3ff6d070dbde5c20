"""The line that bench.py prints on standard output: every key of the contract, and short."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_short_line_keeps_the_contract_and_drops_the_rest():
    import bench
    lat = {"p50": 1.5, "p99": 2.5, "mean": 1.7, "n": 100, "note": "x" * 300}
    table = [{"n_crit": k, "ms": 1.0 / 3, "shape": list(range(20))} for k in range(60)]
    sec = {"value": 1e10 / 3, "block_steps_per_s": 1e4 / 3, "block_step_latency_us": lat, "request_latency_s": lat,
           "by_live": table, "note": "y" * 500, "workload": "z" * 200, "none": None}
    line = {"metric": bench.METRIC, "value": 5e10 / 3, "unit": "interactions/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 50.0 / 3, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded Plummer spheres, seed = rank)",
            "config": {"workload": "w" * 200, "n": 65536, "l2": "flushed (256 MB write) before every timed step"},
            "roofline": {"kernel": "k", "bound": "alu", "achieved": 1.0, "peak": 2.0, "unit": "TFLOP/s", "frac": 0.5,
                         "traffic": 1000, "traffic_capture": "c" * 400, "note": "n" * 900},
            "e2e": {"value": 4e10, "unit": "interactions/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
            "gpu_launches": 123, "tuning": {"fp64": {"candidates": table}}, "active_per_tile": {"counts": table},
            "mixed": sec, "config3": sec, "config1": {"direct_fp64": {"interactions_per_s": 1.0, "peak": "p" * 200}}, "block_step_latency_us": lat,
            "batched": sec, "serving": sec, "serving_sustained": sec,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "cpu_baseline": {"value": 1.0, "unit": "interactions/s", "cores": 16, "kind": "oracle", "sample": "s" * 300}}
    out = bench.short_line(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert out[k] == line[k], k
    assert out["roofline"] == {k: line["roofline"][k] for k in ("kernel", "bound", "achieved", "peak", "unit", "frac", "traffic")}
    assert out["block_step_latency_us"] == out["mixed"]["block_step_latency_us"] == {"p50": 1.5, "p99": 2.5}
    assert abs(out["mixed"]["value"] / sec["value"] - 1.0) < 1e-5
    assert out["config1"] == {"direct_fp64": 1.0}
    assert out["cpu_baseline"] == {"value": 1.0, "unit": "interactions/s", "cores": 16, "kind": "oracle"}
    assert len(json.dumps(out)) < 3000 and json.loads(json.dumps(out)) == out
