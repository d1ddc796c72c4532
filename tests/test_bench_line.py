"""The line bench.py prints: every key a reader needs, short enough to survive in the tail of a log."""
import json

import bench


def _record():
    stat = 1234567.123456789
    entry = {"workload": "llama", "k": {"min": 1, "median": 70.0, "p99": 181.0, "max": 250, "experts_used": 344}, "dense": {str(i): stat for i in range(40)}}
    return {
        "metric": bench.METRIC, "value": stat * 4, "unit": bench.UNIT, "n_gpus": 8, "steps": 1000, "warmup": 100, "ms_per_step": 1.6172123456789012,
        "ms_median": 1.6172123456789012, "ms_min": 1.6, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16 (expert weights e4m3 + 2^k per expert)", "data": "synthetic",
        "config": bench.config_dict(__import__("paper_2310_04361_b200.workloads", fromlist=["CONFIGS"]).CONFIGS["llama"], 0.4, 0.123456789),
        "run": {"tokens_per_gpu": 8192, "k": entry["k"], "l2": "flushed between steps (256 MiB written outside the events)",
                "parallelism": "token-sharded replicas x8, no collective"},
        "e2e": {"value": stat * 3, "unit": bench.UNIT, "h2d_bytes_per_step": 67108864, "d2h_bytes_per_step": 67108864, "ms_median": 2.2771234567,
                "note": "n" * 300},
        "gpu_launches": 9000,
        "roofline": {"bound": "tensor", "kernel": "moe_gather_ffn_kernel (d2d_moe_ffn_fwd, fused path; includes the accumulator's fill and conversion)",
                     "achieved": 333.1234567890123, "peak": 1633.3, "unit": "TFLOP/s", "frac": 0.2039123456789, "executed_frac": 0.5861234567,
                     "traffic": 3019680256, "path_taken": "gather", **{f"x{i}": stat for i in range(20)}},
        "cpu_baseline": {"value": 250.73670690454472, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 200},
        "clocks": {"sm_mhz": 1327.0, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 212},
        "dense_ffn": {"step_interleaved_ms": 1.6172123456789, "torch_eager_ms": 1.7, "library_layer_tau0_ms": 1.6, "speedup_is": "s" * 100},
        "per_config": [entry] * 20}


def test_the_line_is_short_and_complete(capsys, tmp_path):
    record = _record()
    bench.emit(record, None)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 2000
    line = json.loads(out)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                "config"):
        assert line[key] == record[key]
    assert line["value"] > 0 and line["gpu_launches"] == 9000
    assert line["run"]["l2"] == record["run"]["l2"]
    assert set(line["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert set(line["clocks"]) >= {"sm_mhz", "sm_max_mhz", "reasons"}
    assert {"bound", "achieved", "peak", "frac"} <= set(line["roofline"]) and line["cpu_baseline"]["kind"] == "oracle"
    assert json.loads(err) == record                      # nothing is lost: the full record is on stderr
    path = tmp_path / "details.json"
    bench.emit(record, str(path))
    assert json.loads(path.read_text()) == record and capsys.readouterr().err == ""
    record["e2e"] = record["cpu_baseline"] = None         # runs that leave these out
    assert bench.headline(record)["e2e"] is None
