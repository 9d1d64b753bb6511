"""The benchmark's line on standard output stays short whatever its report holds, and keeps what a reader of it needs."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _report():
    return {"metric": bench.METRIC, "value": 1234.5678901234567, "unit": "TFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 3.2123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic",
            "config": {"workload": bench.WORKLOADS[5], "batch_per_gpu": 256, "stack": "x" * 400, "flops": "y" * 100, "l2": "z" * 200},
            "ms_per_step_spread": {k: 3.1234567 for k in ("median", "min", "max", "p10", "p90")} | {"regions": 30},
            "images_per_s": 81234.123456789, "x_dense": 1.2345678901, "ms_per_step_dense": 4.1234567890123,
            "images_per_s_dense": 65432.123456789, "gpu_launches": 33000, "gpu_launches_per_step": 55, "gpu_launches_per_e2e_step": 55,
            "roofline": {"bound": "hbm", "kernel": "k" * 90, "achieved": 1.123456789e3, "peak": 2.0e3, "unit": "TFLOP/s", "frac": 0.5,
                         "how": "h" * 300, "traffic": None, "traffic_note": "n" * 300, "peak_source": "p" * 200},
            "per_layer": [{"layer": f"layer_{i}", "us": 1.0 + i, "note": "l" * 50} for i in range(60)],
            "e2e": {"value": 700.123456789, "unit": "TFLOP/s", "h2d_bytes_per_step": 77070336, "d2h_bytes_per_step": 51380224,
                    "ms_per_step": 5.9876543, "path": "q" * 200},
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "samples": 200, "samples_under_load": 40, "reasons": ["sw_power_cap"],
                       "legs": {f"leg_{i}": {"sm_mhz": 1965.0, "samples": 20, "reasons": ["sw_power_cap"]} for i in range(8)}},
            "dev_status": 0,
            "summary_cfg2": {"rows": list(range(500))},
            "cpu_baseline": {"value": 0.01038, "unit": "TFLOP/s", "cores": 16, "kind": "oracle", "sample": "s" * 300, "images_per_s": 1.2}}


def test_line_is_short_and_complete(capsys):
    report = _report()
    bench.print_line(report)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 2000
    line = json.loads(out)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "gpu_launches", "dev_status"):
        assert line[key] == report[key]
    assert line["config"]["workload"] == report["config"]["workload"]
    assert all(line["clocks"][k] == report["clocks"][k] for k in ("sm_mhz", "sm_max_mhz", "reasons"))
    for key in ("unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == report["e2e"][key]
    assert abs(line["e2e"]["value"] / report["e2e"]["value"] - 1) < 1e-5
    assert json.loads(err)["report"] == report
