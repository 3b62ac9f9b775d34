"""bench.py prints one short line with the fields of its contract, whatever a run
recorded besides; the whole record goes to a file."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_headline_is_short_and_whole(tmp_path, capsys):
    record = {"metric": bench.METRIC, "value": 1.9e8, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
              "ms_per_step": 13.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64",
              "data": "synthetic", "config": {"workload": "scale"}, "roofline": {"bound": "alu"}, "clocks": {},
              "e2e": {"value": 1.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
              "gpu_launches": 7, "serving": {"p50": ["x" * 100] * 300}, "next": {"a": "y" * 20000}}
    bench.emit(record, str(tmp_path / "detail.json"))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 4096
    line = json.loads(out)
    assert line.pop("detail") == "detail.json"
    assert line == {k: v for k, v in record.items() if k not in ("serving", "next")}
    assert json.loads((tmp_path / "detail.json").read_text()) == record
