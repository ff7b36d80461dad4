"""The benchmark's result line: short enough for whoever keeps the end of its output, the tables in a file on demand."""
import json
import os
import sys
import types

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_tables_leave_the_line(tmp_path, capsys):
    sys.path.insert(0, ROOT)
    import bench
    line = {"metric": "m", "value": 1.5, "detail": {"per_dp": list(range(9000))}, "device_status": 0}
    bench.emit(line, types.SimpleNamespace(detail=None))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and json.loads(out) == {"metric": "m", "value": 1.5, "device_status": 0}
    path = tmp_path / "detail.json"
    bench.emit(line, types.SimpleNamespace(detail=str(path)))
    assert json.loads(capsys.readouterr().out)["value"] == 1.5
    assert json.loads(path.read_text()) == line
