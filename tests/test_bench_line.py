"""The benchmark's output line: all that its readers need, and short, however much the record holds."""
import json
import os


def test_line_is_short_and_the_file_holds_everything(tmp_path):
    import bench
    text = "x" * 400
    record = {k: 1.0 for k in bench.LINE_KEYS}
    record["config"] = {"workload": text, "step": text}
    record["e2e"] = {"value": 81.1, "unit": "attempts/ns", "h2d_bytes_per_step": 4096, "d2h_bytes_per_step": 4096}
    record["roofline"] = {"achieved": 2.4, "peak": 40.3, "frac": 0.06, "traffic_basis": text}
    record["clocks"] = {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []}
    record["cpu_baseline"] = {"value": 0.2, "sample": text}
    record["extras"] = {f"workload{k}": {"taus": list(range(2000))} for k in range(8)}
    record["iteration_phase"] = {"ms": [1.0] * 1000}
    out = tmp_path / "sub" / "bench.json"
    printed = bench.output_line(record, out)
    assert "\n" not in printed and len(printed) < 3000
    line = json.loads(printed)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert line[key] == record[key]
    assert json.loads(out.read_text()) == record
    assert line["details"] == os.path.relpath(out)
