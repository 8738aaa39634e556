"""The benchmark's line on stdout: one line of JSON with the keys its readers use,
short enough for a log's tail.  CPU only."""
import json

import bench


def test_the_result_line_is_short_and_complete():
    long = "x" * 5000
    full = {
        "metric": bench.METRIC, "value": 95506338.45362729, "unit": bench.UNIT, "n_gpus": 8, "steps": 100,
        "warmup": 10, "ms_per_step": 10.979124704996744, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "point_mass_2d n=4 m=2 T=1048576 K=4 t=[0,100] X,r per RK4 half-step", "T": 1048576,
                   "n": 4, "m": 2, "K": 4, "l2": "inputs larger than L2 (1.35 GB of coefficient samples)",
                   "parallelism": "replicas x8"},
        "gpu_launches": 135,
        "roofline": {"bound": "alu", "kernel": "build_kernel<4,2> (stage a, with its prepare/terminal launches)",
                     "achieved": 1.8145259038471968, "peak": 1.25856, "unit": "TFLOP/s", "frac": 1.441747635271419,
                     "traffic": None, "peak_source": long},
        "roofline_step": {"note": long},
        "e2e": {"value": 69687863.533567, "unit": bench.UNIT, "h2d_bytes_per_step": 1350566472,
                "d2h_bytes_per_step": 226492640},
        "sequential_gpu": {"value": 4841.066908125368, "unit": bench.UNIT, "T_timed": 16384,
                           "speedup_parallel_over_sequential": 19728.36572312749, "sample": long},
        "pipes_measured": {"how": long},
        "cpu_baseline": {"value": 123596.8813785043, "unit": bench.UNIT, "cores": 1, "sample": long},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 2},
        "rows": {"a4_batched": long},
    }
    text = json.dumps(bench.result_line(full))
    assert len(text) < 2000 and "\n" not in text
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches", "e2e", "clocks"):
        assert json.loads(text)[k] == full[k], k
    full["sequential_gpu"] = full["cpu_baseline"] = None
    assert bench.result_line(full)["sequential_gpu"] is None
