"""The benchmark's stdout line holds the headline and stays short; the secondary measurements go to the detail (CPU
only)."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEADLINE = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline")


def test_line_is_short_and_nothing_is_lost():
    spec = importlib.util.spec_from_file_location("bench_line_mod", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    full = {k: "x" * 100 for k in HEADLINE}
    full["config"] = {"workload": "channel2d_l6", "text": "x" * 400}
    for k in b.DETAIL_KEYS:
        full[k] = {"rows": [1.0] * 500}
    full["fp64_path"] = {"value": 1.5, "ms_per_step": 600.0, "steps": 5, "rtol": 1e-8, "error_vs_oracle": 1e-11,
                         "kernel_classes": {"rows": [1.0] * 500}}
    full["cpu_baseline"] = {"value": 0.01, "unit": "solves/s", "cores": 1, "kind": "oracle", "sample": "x" * 200,
                            "detail": {"rows": [1.0] * 100}, "all_cores": {"value": 0.02}}
    line, detail = b.split_line(full)
    assert len(json.dumps(line)) <= 4096
    assert all(line[k] == full[k] for k in HEADLINE)
    assert line["fp64_path"]["value"] == 1.5 and line["cpu_baseline"]["cores"] == 1
    assert {k: detail.get(k, line.get(k)) for k in full} == full
    poisson = {"solves_per_s": 6.0, "p50_ms": 250.0, "p99_ms": 3000.0, "requests": 256, "failed_instances": [[1.0]] * 99}
    line, detail = b.split_line({"value": 1.0, "served": {"mixed": {"poisson": poisson}}})
    assert line["served"] == {k: v for k, v in poisson.items() if k != "failed_instances"}
    assert detail["served"]["mixed"]["poisson"] == poisson
    line, detail = b.split_line({"value": 1.0, "served": {"error": "x"}})
    assert line == {"value": 1.0} and detail == {"served": {"error": "x"}}
    line, detail = b.split_line({"value": 1.0, "cpu_baseline": None})
    assert line == {"value": 1.0, "cpu_baseline": None} and detail == {}
