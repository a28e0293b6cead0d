"""The line that bench.py prints: every field, and short enough for a reader of the last few thousand characters of the output."""

import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_the_line_is_whole_and_short():
    third = 1234.56789012345678 / 3
    kernels = {f"kernel_class_{i}": {"ms_per_iter": third, "launches_per_iter": third, "gbs": third, "tflops": third,
                                     "roof_ms_per_iter": third, "frac": third} for i in range(14)}
    rec = {"workload": "w" * 200, "value": third, "unit": bench.UNIT, "steps": 20, "warmup": 5, "ms_per_step": third,
           "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap", "gpu_idle"], "samples": 40, "power_w_max": third},
           "gpu_launches": 12345, "t_roof_ms": third, "frac_t_roof": third, "t_roof_note": "n" * 300, "kernels": kernels, "spmm": None,
           "roofline": {"bound": "tensor", "achieved": third, "peak": third, "unit": "TFLOP/s", "peak_source": "p" * 60, "frac": third,
                        "frac_issued": third, "note": "n" * 100, "kernel": "gemm_gradp", "traffic": None},
           "e2e": {"value": third, "unit": bench.UNIT, "h2d_bytes_per_step": third, "d2h_bytes_per_step": third, "note": "n" * 200},
           "cpu_baseline": {"value": third, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 300}, "objective": third}
    workloads = {name: rec for name in bench.ALL}
    workloads["c5"] = {"error": "e" * 1000}
    line = json.dumps(bench.summary_line(rec, workloads, 1, 5, "weak", {"workload": "w" * 200, "parallelism": "p" * 30, "l2": "l" * 80}, 100.0))
    assert len(line) < 4000 and "\n" not in line
    back = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "config", "clocks", "e2e", "gpu_launches", "roofline"):
        assert key in back
    assert set(back["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert abs(back["value"] - third) < 1e-3 and set(back["workloads"]) == set(bench.ALL)
