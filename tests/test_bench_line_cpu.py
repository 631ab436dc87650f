"""The benchmark's output: standard output holds one line, the headline, whatever the side
measurements amount to; these are one JSON object on standard error."""
import ast
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_headline_alone_on_standard_output(capsys):
    sys.path.insert(0, ROOT)
    import bench

    line = {"metric": "m", "value": 1.0, "e2e": {"value": 2.0}, "clocks": {"reasons": []}}
    side = {"batched": {str(i): float(i) for i in range(5000)}, "clean": None}
    bench.print_result(line, side)
    out, err = capsys.readouterr()
    assert out.endswith("\n") and out.count("\n") == 1 and json.loads(out) == line
    assert json.loads(err.strip().splitlines()[-1]) == {"side_measurements": side}


def test_side_measurements_are_not_in_the_headline():
    """The dict literal of the line that main() prints: the contract's keys and no side object."""
    tree = ast.parse(open(os.path.join(ROOT, "bench.py")).read())
    main = next(n for n in tree.body if isinstance(n, ast.FunctionDef) and n.name == "main")
    keys = [[k.value for k in n.value.keys if isinstance(k, ast.Constant)] for n in ast.walk(main)
            if isinstance(n, ast.Assign) and isinstance(n.value, ast.Dict) and getattr(n.targets[0], "id", "") == "line"]
    assert keys == [["metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                     "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks"]]
