"""The default benchmark line runs no configuration that is on record as stalling the GPU."""
import ast
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_serving_block_runs_on_request_only():
    tree = ast.parse(open(os.path.join(ROOT, "bench.py")).read())
    options = {}
    for c in ast.walk(tree):
        if isinstance(c, ast.Call) and getattr(c.func, "attr", "") == "add_argument" and "serving-block" in c.args[0].value:
            options[c.args[0].value] = {k.arg: ast.literal_eval(k.value) for k in c.keywords
                                        if k.arg in ("action", "dest", "default")}
    assert options["--serving-block"] == {"action": "store_true"}
    assert options["--no-serving-block"] == {"action": "store_false", "dest": "serving_block", "default": False}
