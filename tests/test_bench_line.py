"""bench.py's line: headline values as measured, other floats to six digits."""
import bench


def test_short_line():
    x = 1234567.891234567
    line = {"metric": "m", "value": x, "n_gpus": 1, "ms_per_step": x, "vs_baseline": None, "e2e": {"value": x},
            "parts": {"a": x, "b": [x, 3, "t"], "c": {"d": 2.0 / 3}}, "ok": True, "bad": float("inf")}
    got = bench.short_line(line)
    assert list(got) == list(line)
    for k in ("metric", "value", "n_gpus", "ms_per_step", "vs_baseline", "e2e", "ok", "bad"):
        assert got[k] == line[k]
    assert got["parts"] == {"a": 1234570.0, "b": [1234570.0, 3, "t"], "c": {"d": 0.666667}}
