"""The default benchmark line runs no configuration that is on record as stalling the GPU, and its
roofline names the kernel that ran."""
import ast
import os
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_the_serving_block_runs_on_request_only():
    tree = ast.parse(open(os.path.join(ROOT, "bench.py")).read())
    options = {}
    for c in ast.walk(tree):
        if isinstance(c, ast.Call) and getattr(c.func, "attr", "") == "add_argument" and "serving-block" in c.args[0].value:
            options[c.args[0].value] = {k.arg: ast.literal_eval(k.value) for k in c.keywords
                                        if k.arg in ("action", "dest", "default")}
    assert options["--serving-block"] == {"action": "store_true"}
    assert options["--no-serving-block"] == {"action": "store_false", "dest": "serving_block", "default": False}


@pytest.mark.parametrize("layout,D1,D2,B,tile,launches,kernel,bound", [
    (0, 4096, 512, 32, 0, 2.0, "gemm_digit", "tensor"), (0, 4096, 512, 1, 7, 1.0, "scan_tma", "hbm"),
    (0, 100, 16, 2, 9, 1.0, "gemm_digit", "tensor"), (0, 127, 16, 6, 0, 1.0, "gemm_digit", "tensor"),
    (0, 16, 16, 1, 0, 1.0, "scan_direct", "hbm"), (0, 16, 16, 1, 7, 1.0, "scan_direct", "hbm"),
    (0, 64, 512, 32, 6, 1.0, "gemm_plain", "alu"), (0, 512, 256, 1, 1, 1.0, "gemv_scan", "hbm"),
    (1, 512, 256, 32, 0, 1.0, "gemm_digit_limb", "tensor"), (2, 4096, 512, 32, 0, 4.0, "gemm_tc", "tensor"),
])
def test_roofline_kernel(layout, D1, D2, B, tile, launches, kernel, bound):
    import paper_2606_11536_gb300 as g
    from paper_2606_11536_gb300 import build
    build.build()
    ctx = types.SimpleNamespace(g=g, wl="none", peaks={"hbm_gbs": 6800.0}, peak_kind="test", probe=lambda *a: 150.0)
    p = types.SimpleNamespace(n=4096, D1=D1, D2=D2)
    r = bench.gemm_roofline(ctx, layout, B, p, tile, 1.0, launches, {}, None)
    assert (r["kernel"], r["bound"]) == (kernel, bound) and r["frac"] > 0
