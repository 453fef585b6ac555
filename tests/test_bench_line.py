"""bench.py's JSON line stays short enough to survive a reader that keeps the end
of the output, whatever the number of rows behind it."""
import json

import bench


def test_contract_line_is_short():
    rows = [{"level": k, "bound_holds": True, "d": [1.0] * 200} for k in range(11)]
    points = [{"variant": v, "path_steps_per_s": 1e11 / 3 * (1 + k), "ms": 0.1} for k in range(500) for v in ("a", "b")]
    run = {"s_median": 0.00213456789, "prices": [10.4505] * 500, "L": 9, "N": [[1, 2]] * 500, "rms_err_over_eps": 1 / 3}
    out = {"metric": bench.METRIC, "value": 8e11 / 7, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
           "e2e": {"value": 1e11 / 7, "unit": bench.UNIT}, "gpu_launches": 20,
           "bitwidth_optimiser": {"paths_per_level": 10, "levels": rows, "variables": ["Z"] * 100},
           "nested_step_optimised_widths": {"default_formats": {"ms_per_step": 0.1, "var_corrections_euro": [0.1] * 999}},
           "time_to_eps": dict({"m%d" % k: run for k in range(21)}, eps=1e-3, **{"speedup_%d" % k: 1 / 3 for k in range(99)}),
           "sweep_levels": {"scheme": "milstein", "rows": points},
           "serving_sample": [{"requests": 200, "p99_latency_s": 1 / 3, "bias": [1] * 999, "graph_captures": 2}] * 3}
    line = bench.contract_line(out)
    assert len(json.dumps(line)) < 4000 < len(json.dumps(out))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "e2e", "gpu_launches"):
        assert line[k] == out[k]
    assert line["bitwidth_optimiser"]["bounds_hold"] == 11 and line["time_to_eps"]["m3"] == [0.002135, 0.3333]
    assert line["sweep_levels"]["path_steps_per_s"]["a"] == [3.333e10, 1.667e13]
    assert line["serving_sample"][0]["p99_latency_s"] == 0.3333
