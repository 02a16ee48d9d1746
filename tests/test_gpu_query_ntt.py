"""Queries transformed straight into the GEMMs' digits, on the GPU.

From 4096 rows (queries x ciphertexts x components x primes) on, the digit GEMMs' operand is written
by the forward NTT itself.  The plain layout's answers are compared with those of a CUDA-core
tile, which reads NTT-form residues, the limb layout's with its INT8 tile's, and the tensor
layout's with the plain layout's; test_gpu_answer.py compares those with the oracle.  Shapes:
just below and at the line, ciphertext counts that end inside a group of eight and of 64, odd batches
(padded query rows), chunks, every ring.  Residues are whole numbers: equal.
"""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu


def instance(n, L, D1, D2, B):
    p = g.pir_make_params(n, 8, D1, D2, L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(D1 * 100 + B)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    q = torch.empty(B, D1, 2, L, n, dtype=torch.int32, device="cuda")
    for j, prime in enumerate(p.qs):
        q[..., j, :] = torch.randint(0, prime, (B, D1, 2, n), generator=gen, dtype=torch.int32, device="cuda")
    return p, raw, q


def answer(p, raw, q, layout, tile, k_chunk=0):
    db = g.pir_setup_db(p, raw, layout=layout)
    try:
        r = torch.empty(q.shape[0], p.D2, 2, p.L, p.n, dtype=torch.int32, device="cuda")
        g.pir_answer_ex(db, q, q.shape[0], r, tile=tile, k_chunk=k_chunk)
        torch.cuda.synchronize()
        g.pir_check_device()
        return r
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("n,L,D1,D2,B,k_chunk", [
    (2048, 2, 128, 32, 8, 0), (2048, 1, 255, 24, 8, 0), (2048, 3, 233, 20, 3, 0), (2048, 2, 130, 32, 33, 0),
    (4096, 2, 261, 16, 5, 0), (4096, 1, 2047, 8, 2, 0), (4096, 4, 129, 12, 7, 0), (8192, 2, 135, 8, 9, 0),
    (8192, 3, 512, 4, 2, 0), (4096, 2, 420, 16, 5, 209), (2048, 2, 64, 16, 17, 0)])
def test_plain(n, L, D1, D2, B, k_chunk):
    p, raw, q = instance(n, L, D1, D2, B)
    assert torch.equal(answer(p, raw, q, g.PIR_LAYOUT_PLAIN, 9, k_chunk), answer(p, raw, q, g.PIR_LAYOUT_PLAIN, 4, k_chunk))


@pytest.mark.parametrize("n,L,D1,D2,B", [(2048, 2, 96, 16, 12), (4096, 2, 288, 32, 5), (8192, 1, 160, 8, 13)])
def test_limb(n, L, D1, D2, B):
    p, raw, q = instance(n, L, D1, D2, B)
    assert torch.equal(answer(p, raw, q, g.PIR_LAYOUT_LIMB, 0), answer(p, raw, q, g.PIR_LAYOUT_LIMB, 1))


@pytest.mark.parametrize("n,L,D1,D2,B", [(2048, 2, 128, 64, 8), (4096, 3, 192, 32, 5), (8192, 2, 64, 32, 17)])
def test_tensor(n, L, D1, D2, B):
    p, raw, q = instance(n, L, D1, D2, B)
    assert torch.equal(answer(p, raw, q, g.PIR_LAYOUT_TENSOR, 0), answer(p, raw, q, g.PIR_LAYOUT_PLAIN, 4))
