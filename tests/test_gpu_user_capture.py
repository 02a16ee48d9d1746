"""Calls captured into the caller's own CUDA graph, each as the first call of a process: nothing
that they need may be allocated in a way that a capture refuses."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import torch
import paper_2606_11536_gb300 as g
gen = torch.Generator(device="cuda")
gen.manual_seed(4)

def words(*shape, lo=-2**31, hi=2**31 - 1, dtype=torch.int32):
    return torch.randint(lo, hi, shape, generator=gen, dtype=dtype, device="cuda")

def captured(call):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph
"""

LWE = HEAD + """
D1, D0, B = 777, 2048, 8
db, qs = words(D1 * D0, lo=-128, hi=128, dtype=torch.int8), [words(B * D0) for _ in range(3)]
q, out, want = torch.empty_like(qs[0]), torch.empty(B * D1, dtype=torch.int32, device="cuda"), None
graph = captured(lambda: g.pir_lwe_answer(db, D1, D0, q, B, out, path=g.PIR_LWE_TENSOR))
for x in qs:
    q.copy_(x)
    out.zero_()
    graph.replay()
    got = out.clone()
    g.pir_lwe_answer(db, D1, D0, x, B, out, path=g.PIR_LWE_SIMT)
    assert torch.equal(got, out)
g.pir_check_device()
"""

ANSWER = HEAD + """
n, L, D1, D2, B = 2048, 2, 128, 64, 4
p = g.pir_make_params(n, 8, D1, D2, L)
db = g.pir_setup_db(p, words(D1 * D2 * n, lo=0, hi=256, dtype=torch.uint8), %s)
qs = [words(B, D1, 2, L, n, lo=0, hi=min(p.qs)) for _ in range(3)]
q, out = torch.empty_like(qs[0]), torch.empty(B * D2 * 2 * L * n, dtype=torch.int32, device="cuda")
graph = captured(lambda: g.pir_answer(db, q, B, out))
for x in qs:
    q.copy_(x)
    out.zero_()
    graph.replay()
    got = out.clone()
    g.pir_answer(db, x, B, out)
    assert torch.equal(got, out)
g.pir_check_device()
g.pir_free_db(db)
"""


@pytest.mark.parametrize("script", [LWE, ANSWER % "g.PIR_LAYOUT_PLAIN", ANSWER % "g.PIR_LAYOUT_LIMB",
                                    ANSWER % "g.PIR_LAYOUT_TENSOR"], ids=["lwe", "plain", "limb", "tensor"])
def test_first_call_of_a_process(script):
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
