"""bench.py's result line keeps the headline's keys and stays below 2 kB, whatever
the details weigh."""
import json

import bench


def test_result_line_is_short_and_complete():
    arms = {"arm%d" % i: {"speedup": 1.0 / 3.0, "iters": list(range(40))} for i in range(100)}
    line = {
        "metric": bench.METRIC, "value": 800.0 / 3.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 10,
        "warmup": 3, "ms_per_step": 59.0 / 3.0, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": bench.WORKLOAD, "method": "plain Jacobi", "grids_per_gpu": 16,
                   "l2": "flushed between steps (256 MB write, untimed)",
                   "iters_per_grid": [5000] * 16},
        "roofline": {"bound": "alu", "kernel": "sweep_resident_kernel", "achieved": 12.0,
                     "peak": 40.0, "unit": "TOP/s", "frac": 0.3, "traffic": 1, "note": "x" * 500},
        "e2e": {"value": 1.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
        "gpu_launches": 60, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
        "hybrid": arms, "driver_step": arms, "stencil_roofline": arms,
        "hybrid_vs_plain": {"best_network_equal_threshold": {"network": "a", "speedup": 1.5},
                            "others": arms}}
    text = json.dumps(bench.result_line(line))
    got = json.loads(text)
    assert len(text) < 2000 and "\n" not in text
    for k in set(line) - {"hybrid", "driver_step", "stencil_roofline"}:
        assert k in got, k
    assert abs(got["value"] / line["value"] - 1.0) < 1e-6
    assert got["e2e"] == line["e2e"] and got["clocks"] == line["clocks"]
    assert "iters_per_grid" in line["config"]
