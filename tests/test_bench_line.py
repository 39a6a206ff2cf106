"""The benchmark's printed line: the keys of its contract, short enough to survive
in the last 3,000 characters of the output, the long sections in a file."""
import json

import bench

KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
        "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline")


def _line():
    line = {k: {"note": "x" * 60, "value": 0.1234567890123456} for k in KEYS}
    line.update({k: [{"some": "x" * 100}] * 50 for k in bench.DETAILS})
    return line


def test_line_is_short_and_keeps_its_keys(tmp_path):
    line, path = _line(), str(tmp_path / "d.json")
    short = bench.headline(line, path)
    assert len(json.dumps(line)) > 20000 and len(json.dumps(short)) < 3000
    assert all(short[k] == line[k] for k in KEYS) and short["details"] == path
    assert json.load(open(path)) == line


def test_line_without_a_place_for_details(tmp_path):
    short = bench.headline(_line(), str(tmp_path / "missing" / "d.json"))
    assert short["details"] is None and all(k in short for k in KEYS)
