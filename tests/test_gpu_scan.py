"""The plain layout's paths by size: the staged and the direct scan, the GEMM tiles and the
digit GEMM, on the GPU.

The default tile, whatever path it takes for a shape, gives what a named CUDA-core tile gives
(the GEMV for one and two queries, the 16 x 256 GEMM tile else), whose own results
test_gpu_answer.py compares with the oracle.  Shapes sit on both sides of the lines between the
paths and at their tiles' edges; K-chunks accumulate.  Residues are whole numbers: equal.
"""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu

# (D1, D2): strips and quads of the direct scan, the staged scan's columns and length
FEW = [(1, 4), (2, 12), (16, 16), (17, 20), (33, 100), (40, 132), (63, 256), (64, 256), (86, 192), (87, 188), (32, 512),
       (64, 512), (72, 448), (73, 444), (130, 260)]
# (D1, D2, B): direct scan, tile and digits by cost; query rows in one, two and many passes
MANY = [(1, 4, 3), (16, 16, 4), (16, 64, 5), (24, 128, 6), (40, 48, 9), (64, 132, 5), (64, 512, 3), (96, 200, 4), (63, 16, 33),
        (16, 256, 17), (16, 24, 64), (127, 32, 12), (128, 16, 3), (127, 256, 8)]


def answers(n, L, D1, D2, B, tiles, k_chunk=0):
    p = g.pir_make_params(n, 8, D1, D2, L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(D1 * 1000 + D2)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    q = torch.empty(B, D1, 2, L, n, dtype=torch.int32, device="cuda")
    for j, prime in enumerate(p.qs):
        q[..., j, :] = torch.randint(0, prime, (B, D1, 2, n), generator=gen, dtype=torch.int32, device="cuda")
    db = g.pir_setup_db(p, raw)
    try:
        out = []
        for tile in tiles:
            r = torch.empty(B, D2, 2, L, n, dtype=torch.int32, device="cuda")
            g.pir_answer_ex(db, q, B, r, tile=tile, k_chunk=k_chunk)
            out.append(r)
        torch.cuda.synchronize()
        g.pir_check_device()
        return out
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("D1,D2", FEW)
@pytest.mark.parametrize("B", [1, 2])
def test_scan_by_size_equals_gemv(D1, D2, B):
    got, scan, want = answers(2048, 1 + D1 % 3, D1, D2, B, (0, 7, B))
    assert torch.equal(got, want)
    assert torch.equal(scan, want)


@pytest.mark.parametrize("D1,D2,B", MANY)
def test_default_path_equals_gemm_tile(D1, D2, B):
    got, want = answers(2048, 1 + D1 % 2, D1, D2, B, (0, 4))
    assert torch.equal(got, want)


@pytest.mark.parametrize("D1,D2,B,k_chunk", [(40, 32, 1, 16), (41, 32, 1, 13), (200, 256, 1, 80), (50, 132, 2, 20),
                                             (60, 16, 5, 25), (60, 48, 9, 44)])
def test_chunks_accumulate(D1, D2, B, k_chunk):
    got, want = answers(2048, 2, D1, D2, B, (0, 4), k_chunk)
    whole, = answers(2048, 2, D1, D2, B, (0,))
    assert torch.equal(got, want)
    assert torch.equal(got, whole)
