"""The benchmark's own line stays short: the studies beside it (some 20 KB of JSON) go to stderr,
so that the line can be read whole from the last 4 KB of a log (no GPU)."""
import ast
import json
import os

import bench

STUDIES = {"other_workloads", "coexistence", "interface", "stability", "calibration", "dynamics",
           "batch_equilibrium", "precision_error", "warm_start"}


def test_studies_are_no_part_of_the_line():
    tree = ast.parse(open(os.path.abspath(bench.__file__)).read())
    keys = {n.slice.value for n in ast.walk(tree)
            if isinstance(n, ast.Subscript) and isinstance(n.ctx, ast.Store)
            and isinstance(n.value, ast.Name) and n.value.id == "line"}
    assert keys <= {"cpu_baseline", "roofline_fp64"}, keys
    names = {n.value for n in ast.walk(tree) if isinstance(n, ast.Constant)}
    assert STUDIES <= names  # and each is still reported


def test_report_prints_to_stderr_and_hides_no_error(capsys):
    bench.report("study", lambda a: {"value": a}, 3)
    bench.report("broken", lambda: 1 / 0)
    out, err = capsys.readouterr()
    assert out == ""
    rows = dict(line.split(": ", 1) for line in err.splitlines())
    assert json.loads(rows["study"]) == {"value": 3}
    assert "ZeroDivisionError" in json.loads(rows["broken"])["error"]
