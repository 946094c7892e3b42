"""The line bench.py prints on stdout stays a few kB long whatever was measured (a reader may keep only the end of
the output), holds the keys of its contract, and its figures are those of the full record, which goes to stderr
before it."""
import json
import os
import types

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
        "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline", "roofline")


def _record():
    with open(os.path.join(ROOT, "profiles", "bench__wake_2048x256_m2_fp64.json")) as f:
        return json.load(f)


def test_default_run(capsys, tmp_path):
    r = _record()
    assert len(json.dumps(r)) > 15000   # the other forms, the large run and 64 scan members among it
    bench.emit(r, types.SimpleNamespace(record=str(tmp_path / "r.json")))
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.LINE_BYTES + 1
    line = json.loads(out)
    for k in KEYS:
        assert k in line, k
    for k in ("value", "ms_per_step", "e2e", "gpu_launches", "steps", "warmup"):
        assert line[k] == r[k], k
    assert line["config"] == r["config"] and line["clocks"] == r["clocks"]
    assert abs(line["scan"]["value"] / r["scan"]["value"] - 1) < 1e-5
    assert json.loads(err.split("record: ", 1)[1]) == r
    assert json.loads((tmp_path / "r.json").read_text()) == r


def test_scan_of_many():
    r = _record()["scan"]
    r["config"].update({k: list(range(1000)) for k in ("Nz", "Nr", "Nm", "order_p", "band_chunk")})
    line = bench.short_line({**r, "metric": "pic_steps_per_s"})
    assert len(line) <= bench.LINE_BYTES
    assert json.loads(line)["config"]["Nz"] == {"n": 1000, "min": 0, "max": 999}


def test_what_is_too_long_is_left_out():
    r = _record()
    r["chosen_form"]["criterion"] = "x" * 5000
    line = bench.short_line(r)
    assert len(line) <= bench.LINE_BYTES
    assert all(k in json.loads(line) for k in KEYS)
