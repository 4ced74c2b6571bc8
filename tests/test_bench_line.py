"""The benchmark's output: one JSON line on stdout that stays short whatever the legs report."""
import json


def test_legs_go_to_stderr(capsys):
    import bench
    line = {"metric": bench.METRIC, "value": 1.5, "e2e": {"value": 1.0}}
    bench.emit(line, {"serving": {str(i): "x" * 100 for i in range(500)}})
    out, err = capsys.readouterr()
    assert json.loads(out) == line and out.count("\n") == 1
    assert len(json.loads(err)["legs"]["serving"]) == 500
    bench.emit(line, {})
    assert capsys.readouterr().err == ""


def test_the_line_takes_no_legs():
    import inspect

    import bench
    src = inspect.getsource(bench.run_ours)
    assert "line.update(" not in src and "print(" not in src
