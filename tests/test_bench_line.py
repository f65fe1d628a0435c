"""The benchmark's one line on standard output stays short whatever sections a run has."""
import json

import bench


def test_sections_go_to_standard_error_and_the_line_keeps_its_keys(capsys):
    keys = ["metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
            "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"]
    out = {k: 1.5 for k in keys}
    out["sweep"] = [{"workload": "x" * 100, "ms": 1.0}] * 200
    out["lazy_update"] = {"rows": ["y" * 100] * 50}
    bench.report(out)
    got = capsys.readouterr()
    assert got.out.count("\n") == 1
    line = json.loads(got.out)
    assert line == {k: 1.5 for k in keys}
    sections = [json.loads(x) for x in got.err.splitlines()]
    assert [s["section"] for s in sections] == ["sweep", "lazy_update"]
    assert sections[0]["sweep"] == out["sweep"]
