"""The benchmark's printed line: every key of its contract, on one line, short
enough to survive in the last kilobytes of a program's output whatever the
legs add to the record."""
import json

import pytest

bench = pytest.importorskip("bench")

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline")


def record():
    r = {k: 1.0 for k in bench.LINE_KEYS}
    r["config"] = dict(bench.WORKLOAD, note="n" * 300)
    r["roofline"] = {"kernel": "k" * 1400}
    r["cpu_baseline"] = {"sample": "s" * 600}
    for leg in ("pcg", "three_d", "batched", "redistribution", "threshold_sweep"):
        r[leg] = {"workload": "w" * 100, "fp64": {"value": 2.0}, "rows": [{"x": i} for i in range(2000)]}
    r["redistribution"] = {"rows": list(range(5000))}
    return r


@pytest.mark.parametrize("to_file", [True, False])
def test_line_is_short_and_whole(to_file, tmp_path, capsys):
    r = record()
    path = tmp_path / "record.json"
    bench.write_record(r, str(path) if to_file else None)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 6000
    line = json.loads(out)
    assert all(k in line for k in CONTRACT)
    assert line["value"] == r["value"]
    assert line["legs_unknowns_per_s"]["pcg"] == 2.0 and "redistribution" not in line["legs_unknowns_per_s"]
    assert json.loads(path.read_text() if to_file else err) == r
