"""The benchmark's line on stdout: every key that is read from it, in a length that survives where only the end of the output is kept."""
import json


def test_headline_is_short_and_complete():
    import bench
    big = [{"note": "x" * 400}] * 60
    out = {"metric": bench.METRIC, "value": 34878.297057939075, "unit": bench.UNIT, "n_gpus": 1, "steps": 200, "warmup": 5, "ms_per_step": 1.8349519729614259,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "tf32", "data": "synthetic",
           "config": {"workload": "resnet50_conv_stack_b64_224_2of4", "layers": 53, "batch_per_gpu": 64, "tile_t": 64, "plans": "per layer by nm_autotune",
                      "cache": "inputs larger than L2 (5.4 GB touched per step, one buffer per layer)", "parallelism": "replicas x1"},
           "useful_tflops": 145.78929609911862, "gpu_launches": 10600, "stack_roofline_frac": 0.4912345678901234,
           "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 12},
           "e2e": {"value": 1003.123456789, "unit": bench.UNIT, "h2d_bytes_per_step": 2790000000, "d2h_bytes_per_step": 2790000000, "note": "x" * 200},
           "roofline": {"bound": "hbm", "achieved": 3300.123456789, "peak": 6532.9, "unit": "GB/s", "frac": 0.5051612345678, "traffic": 123456789.123, "kernel": "k_conv_expand",
                        "note": "x" * 300},
           "gather_only": {"value": 34669.22437675706, "note": "x" * 300}, "chained": {"value": 34878.297057939075, "note": "x" * 300},
           "parity": {"ok": True, "layers": big}, "cpu_baseline": {"value": 1.4784184219167196, "unit": bench.UNIT, "cores": 128, "sample": big},
           "per_layer": big, "tile_choice": big}
    line = json.dumps(bench.headline(out))
    assert len(line) < 1450
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                "config", "gpu_launches", "clocks", "e2e", "roofline"):
        assert key in got
    assert got["value"] == out["value"] and set(got["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
