"""The measurements of bench.py outside the timed step take the step's own inputs:
none of its functions gives a parameter another value on the way (the drift search's
channel axis once took the place of the sky frequencies, and the imaging below it ran
at 0 to 511 Hz)."""
import ast
import inspect

import bench


def test_no_function_rebinds_a_parameter():
    tree = ast.parse(inspect.getsource(bench))
    seen = 0
    for f in ast.walk(tree):
        if isinstance(f, ast.FunctionDef):
            args = {a.arg for a in f.args.posonlyargs + f.args.args + f.args.kwonlyargs}
            stored = {n.id for n in ast.walk(f) if isinstance(n, ast.Name) and isinstance(n.ctx, ast.Store)}
            assert not args & stored, (f.name, args & stored)
            seen += f.name == "next_row_measurements"
    assert seen == 1
