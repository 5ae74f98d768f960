"""The line that bench.py prints on stdout stays short: a log that keeps the last 4 KB keeps it whole."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_summary_line_is_short_and_complete():
    sys.path.insert(0, ROOT)
    import bench
    layer = {"layer": "256->256@1024x1024n1", "tile": 4, "us": 977.66, "us_input": 297.62, "us_gemm": 415.63, "us_output": 264.41,
             "us_fused": 0.0, "eq_tflops": 1265.2, "bound": "tensor", "roof_us": 188.24, "frac_of_roof": 0.193, "gemm_tensor_frac": 0.453}
    e2e = {"value": 123.45, "unit": "TFLOP/s", "h2d_bytes_per_step": 10 ** 9, "d2h_bytes_per_step": 10 ** 9, "api": "x" * 250}
    clocks = {"sm_mhz": 1965, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 33}
    roofline = {"kernel": "wino_gemm_kernel", "bound": "tensor", "achieved": 1, "peak": 2, "unit": "TFLOP/s", "frac": 0.5,
                "peak_source": "y" * 200, "traffic": None, "traffic_source": "z" * 200, "launches_per_step": 25.0}
    work = {"value": 1000.0, "unit": "TFLOP/s", "ms_per_step": 4.7, "e2e": e2e, "layers": [layer] * 26, "cudnn_yardstick": {"value": 500.0}}
    names = ("single", "sd15_unet", "sd_vae_512", "sd21_unet", "sdxl_1024")
    line = {"metric": bench.metric_name("sdxl_1024"), "value": 1000.0, "unit": "TFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 4.7, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f16", "data": "synthetic",
            "config": {"workload": "sdxl_1024", "tile_per_layer": [4] * 26, "algorithm": "a" * 200, "l2": "b" * 200, "step_call": "c" * 60,
                       "filter_transform": "d" * 70, "other_workloads_in_this_line": list(names), "batch": 2},
            "e2e": e2e, "gpu_launches": 1000, "clocks": clocks, "sustained": {"value": 1.0, "ms_per_step": 4.7, "clocks": clocks},
            "roofline": roofline, "transforms": {"input_transform": {"gbs": 1.0}}, "cpu_baseline": {"value": 0.01, "sample": "s" * 700},
            "cudnn_yardstick": {"value": 500.0}, "layers": [layer] * 26, "workloads": {n: dict(work) for n in names}}
    short = bench.summary_line(line)
    assert len(json.dumps(short)) < 4000 < len(json.dumps(line))
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "e2e", "gpu_launches", "clocks"):
        assert short[key] == line[key], key
    assert short["config"]["workload"] == "sdxl_1024" and short["workloads"]["single"]["value"] == 1000.0
    line["sustained"] = line["cpu_baseline"] = line["roofline"] = None          # the switches that skip parts
    line["workloads"] = {"single": {**work, "e2e": None, "cudnn_yardstick": None}}
    assert bench.summary_line(line)["workloads"]["single"]["e2e"] is None
