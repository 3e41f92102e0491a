"""The benchmark's result line stays short enough to be read off the end of a
log; the breakdowns and the other workloads go to a file (no GPU)."""
import json

import bench


def _result():
    layers = {f"layer{i}.conv{i}": [0.123456] * 5 for i in range(54)}
    return {"metric": bench.METRIC, "value": 169.9, "unit": "TOPS", "n_gpus": 1, "steps": 50,
            "warmup": 5, "ms_per_step": 24.6, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u8", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD}, "roofline": {"frac": 0.5},
            "per_call_ms": dict.fromkeys(bench.CALLS, 1.0), "rooflines": {c: layers for c in bench.CALLS},
            "per_layer_ms": layers, "slowest_layers": [layers] * 6, "stem_grad_x_ms": 0.7,
            "clocks": {"sm_mhz": 2070.0}, "gpu_launches": 28300, "device_status": 0,
            "e2e": {"value": 15.8}, "extras": {"a": [layers] * 10}, "cpu_baseline": {"value": 0.04}}


def test_the_line_is_short_and_the_details_are_kept(tmp_path, capsys):
    path = tmp_path / "details.json"
    bench.report(_result(), str(path))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 4096
    line, details = json.loads(out), json.loads(path.read_text())
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "clocks",
              "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert line[k] == _result()[k]
    assert line["details"] == str(path)
    assert {**line, **details} == {**_result(), "details": str(path)}


def test_a_details_file_that_cannot_be_written_costs_no_result(tmp_path, capsys):
    bench.report(_result(), str(tmp_path / "absent" / "details.json"))
    line = json.loads(capsys.readouterr().out)
    assert line["value"] == 169.9 and line["details"].startswith("not written")
