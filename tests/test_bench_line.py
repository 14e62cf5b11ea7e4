"""bench.py's line: one JSON object on stdout, short enough for a reader that
keeps the last few KB of the output; the tables go to stderr."""
import json


def test_line_is_short_and_alone_on_stdout(capsys):
    import bench
    row = {"layer": "l", "shape": "256->256 14x14 k3 s1", "routine": "conv2/igemm_tc " + "x" * 80, "us": 1.0 / 3}
    clk = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 5}
    roof = {"bound": "tensor", "achieved": 1e3 / 3, "peak": 1687.4, "unit": "TFLOP/s", "frac": 2 / 3, "traffic": None,
            "traffic_unit": "u" * 70, "algorithmic_flop": 1 << 40, "algorithmic_bytes": 1 << 40, "share_of_step": 0.9,
            "time_ms": 2 / 3, "method": "m" * 180, "kernel": "conv2/igemm_tc", "peak_source": "measured (MEASURED_PEAKS.json)"}
    line = {"metric": bench.METRIC, "value": 1e5 / 3, "unit": "images/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 2 / 3, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic", "config": {"workload": bench.WORKLOAD, "batch": 32, "parallelism": "replicas x1",
                                            "l2": "l" * 60, "timing": "t" * 80},
            "e2e": {"value": 1e5 / 3, "unit": "images/s", "h2d_bytes_per_step": 9633792, "d2h_bytes_per_step": 64000,
                    "call": "c" * 160}, "gpu_launches": 1260, "roofline": roof,
            "cpu_baseline": {"value": 1.0, "unit": "images/s", "cores": 16, "kind": "oracle", "sample": "s" * 100},
            "clocks": clk, "tuning_s": 20.0, "path_cost_ns": 1, "plan": "tuned in this run",
            "r50_b1_fp16_latency": {"mean_ms": 1 / 3, "std_ms": 1 / 3, "median_ms": 1 / 3},
            "activation_memory": {"arena_bytes": 1}, "per_routine_ms": {}, "per_layer": [row] * 60,
            "extras": {"sweep": {"rows": [row] * 40}}}
    bench.emit(line)
    got = capsys.readouterr()
    assert got.out.count("\n") == 1 and len(got.out) < 2300
    out = json.loads(got.out)
    assert set(out) == set(line) - set(bench.DETAILS)
    assert abs(out["value"] - line["value"]) < 1e-6 * line["value"]
    assert json.loads(got.err)["details"]["per_layer"] == line["per_layer"]
