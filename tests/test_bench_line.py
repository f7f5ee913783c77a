"""The benchmark's one line on stdout: short enough to be kept whole with the end of a run's output, and with every key that
a reader of it needs, whatever the run measured beside them."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_summary_is_short_and_whole():
    import bench
    x = 12345.678901234567
    line = {"metric": bench.METRIC, "value": x, "unit": "updates/s", "n_gpus": 8, "steps": 1000, "warmup": 100, "ms_per_step": x / 1e5,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "n_sites": 4320, "n_charges": 5700, "n_kvectors": 17719, "replicas_per_step": 8,
                       "k_prec": "f16x2", "path": "p" * 300, "parallelism": "replicas x8"},
            "e2e": {"value": x, "unit": "updates/s", "h2d_bytes_per_step": 1459328, "d2h_bytes_per_step": 276544, "path": "q" * 300},
            "gpu_launches": 123456, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 60},
            "fp64_value": x / 7, "speedup_vs_fp64": x / 3e3, "rel_err_mixed_vs_fp64": 2.13070695959304e-06, "max_abs_qtot": 1.3e-15,
            "roofline": {"bound": "alu", "unit": "TFLOP/s", "achieved": x / 700, "kernel": "k_rows_sf<float>", "frac": 1 / 7,
                         "ms_per_launch": x / 1e6, "all_kernels": {str(k): x for k in range(50)}},
            "cpu_baseline": {"value": 1 / 7, "unit": "updates/s", "cores": 16, "kind": "oracle", "sample": "s" * 500},
            "cfg4_serving": {str(k): x for k in range(500)}}
    text = json.dumps(bench.summary(line))
    assert "\n" not in text and len(text) <= bench.SUMMARY_BYTES
    out = json.loads(text)
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                "gpu_launches"):
        assert out[key] == line[key], key
    assert abs(out["value"] / line["value"] - 1.0) < 1e-5 and abs(out["ms_per_step"] / line["ms_per_step"] - 1.0) < 1e-5
    assert out["e2e"]["h2d_bytes_per_step"] == 1459328 and out["e2e"]["d2h_bytes_per_step"] == 276544
    assert out["clocks"]["sm_mhz"] == 2070.0 and out["clocks"]["reasons"] == ["sw_power_cap"]
    assert out["config"]["workload"] == bench.WORKLOAD and out["config"]["replicas_per_step"] == 8
    print(len(text))
