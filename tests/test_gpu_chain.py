"""Kernels that start while their predecessor drains, on the GPU.

Chains of in-place transforms and answers without a synchronization between them, on one and on
two streams and with other kernels of the stream in between: every kernel must see all of what
the one before it wrote.  Transforms there and back give the input again, whole numbers: equal.
"""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu


def residues(p, count, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.empty(count, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, q in enumerate(p.qs):
        x[:, j] = torch.randint(0, q, (count, p.n), generator=gen, dtype=torch.int32, device="cuda")
    return x


# rows: one block, a partial wave, several waves
@pytest.mark.parametrize("n,L,count", [(2048, 1, 1), (4096, 2, 97), (8192, 3, 301), (4096, 2, 3000)])
def test_transforms_in_place(n, L, count):
    p = g.pir_make_params(n, 8, 1, 1, L)
    x = residues(p, count, n)
    want = x.clone()
    for _ in range(20):
        g.ntt_fwd(p, x)
        g.ntt_inv(p, x)
    assert torch.equal(x, want)
    for _ in range(10):  # other kernels of the stream between the transforms
        g.ntt_fwd(p, x)
        y = x.clone()
        x.zero_()
        g.ntt_inv(p, y)
        x.copy_(y)
    assert torch.equal(x, want)


def test_two_streams():
    p = g.pir_make_params(4096, 8, 1, 1, 2)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    xs = [residues(p, 500, s) for s in range(2)]
    want = [x.clone() for x in xs]
    torch.cuda.synchronize()
    for _ in range(20):
        for x, s in zip(xs, streams):
            g.ntt_fwd(p, x, stream=s)
            g.ntt_inv(p, x, stream=s)
    torch.cuda.synchronize()
    for x, w in zip(xs, want):
        assert torch.equal(x, w)


def test_small_answers_back_to_back():
    p = g.pir_make_params(2048, 12, 16, 16, 2)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    raw = torch.randint(0, 256, (16 * 16 * 2048 * 12 // 8,), generator=gen, dtype=torch.uint8, device="cuda")
    db = g.pir_setup_db(p, raw)
    try:
        qs = [residues(p, 32, 10 + k).view(1, 16, 2, 2, 2048) for k in range(8)]
        alone = []
        for q in qs:
            r = torch.empty(1, 16, 2, 2, 2048, dtype=torch.int32, device="cuda")
            g.pir_answer(db, q, 1, r)
            torch.cuda.synchronize()
            alone.append(r)
        q, r = torch.empty_like(qs[0]), torch.empty_like(alone[0])
        got = []
        for k in range(40):  # one query and one response buffer, rewritten between the calls
            q.copy_(qs[k % 8])
            g.pir_answer(db, q, 1, r)
            got.append(r.clone())
        for k, x in enumerate(got):
            assert torch.equal(x, alone[k % 8])
    finally:
        g.pir_free_db(db)
