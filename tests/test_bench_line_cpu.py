"""The line that bench.py prints: short enough to be read whole from the end of a
log, with everything else in the detail file."""
import json

import bench


def full_line():
    return dict({k: 1.0 for k in bench.LINE_KEYS}, metric=bench.METRIC, unit=bench.UNIT,
                config={"workload": "w" * 300, "shape": [1] * 40}, e2e={"value": 2.0, "h2d_bytes_per_step": 3},
                roofline={"kernel": "k" * 200}, cpu_baseline={"value": 4.0, "sample": "s" * 300},
                forms={str(k): {"ms": float(k)} for k in range(2000)}, extensions="x" * 20000)


def test_line_is_short_and_the_file_has_everything(tmp_path):
    line = full_line()
    path = str(tmp_path / "detail.json")
    text = json.dumps(bench.short_line(line, path))
    assert len(text) <= bench.LINE_MOST + 200 and "\n" not in text
    got = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert got[k] == line[k], k
    assert got["detail"] == path and "forms" not in got
    with open(path) as f:
        assert json.load(f) == line


def test_a_line_that_is_too_long_keeps_the_contract(tmp_path):
    line = full_line()
    line["latency_ms"] = {str(k): float(k) for k in range(1000)}
    line["samples_per_s"] = "y" * 9000
    got = bench.short_line(line, str(tmp_path / "no" / "such" / "folder"))   # the line is printed all the same
    assert "detail" not in got and "latency_ms" not in got and "samples_per_s" not in got
    assert got["roofline"] == line["roofline"] and len(json.dumps(got)) <= bench.LINE_MOST
