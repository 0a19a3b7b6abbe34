"""The result line of bench.py: the contract's keys, and short enough to survive a reader that keeps the end of the output."""
import json


def test_the_line_is_short_and_complete():
    import bench
    e2e = {"value": 234.7019801728156, "unit": "GFLOP/s", "ms_per_step": 35.302, "h2d_bytes_per_step": 1612800000, "d2h_bytes_per_step": 6400000}
    per = {str(i): {"ms_per_step": 4.799999123, "execute_ms": 1.099993412, "value_gflops": 1789.123451, "e2e": e2e} for i in range(1, 6)}
    line = {"metric": "useful GFLOP/s", "value": 1821.123456789, "unit": "GFLOP/s", "n_gpus": 8, "steps": 20, "warmup": 5,
            "ms_per_step": 4.6812345, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "ttmc3_skewed_12000x9000x29000_nnz77M_r16", "scale": 1.0, "step": "const_csf_build + const_execute",
                       "nnz": 77000000, "level_sizes": {"X": [12000, 11953580, 77000000]}, "l2": "inputs larger than L2 (no flush)",
                       "replicas": 8, "per_config": per},
            "roofline": {"kernel": "rs_onesweep", "bound": "hbm", "achieved": 3302.12345, "peak": 6548.8, "unit": "GB/s", "frac": 0.4923412,
                         "traffic": 1745000000.0, "peak_source": "measured"},
            "cpu_baseline": {"value": 1.23456789, "unit": "GFLOP/s", "cores": 16, "kind": "oracle", "sample": "x" * 200},
            "max_err_ratio": 0.013987, "e2e": e2e, "gpu_launches": 260, "kernels": [{"name": "rs_onesweep"}] * 40,
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "samples": 6}}
    text = json.dumps(bench.short_line(line))
    assert len(text) < 1300
    out = json.loads(text)
    assert {"metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
            "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"} <= set(out)
    assert abs(out["value"] / line["value"] - 1) < 1e-4 and abs(out["ms_per_step"] / line["ms_per_step"] - 1) < 1e-4
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(out["e2e"])
