"""Expansion and folding levels: two ciphertexts a thread against one, on the GPU.

A batch large enough that the last expansion levels (the first folding levels) take two
ciphertexts a thread gives, query by query, what calls of one query give, whose levels take
one; those are compared with the oracle in test_gpu_expand.py and test_gpu_fold.py.  Residues
are whole numbers: equal, not close.
"""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu


def residues(gen, lead, p):
    out = torch.empty(*lead, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, q in enumerate(p.qs):
        out[..., j, :] = torch.randint(0, q, (*lead, p.n), generator=gen, dtype=torch.int32, device="cuda")
    return out


# (n, L, ell, B, levels, count): counts that end inside and at a thread's pair
EXPAND = [(2048, 1, 2, 40, 5, 32), (4096, 2, 4, 20, 5, 27), (4096, 3, 9, 16, 5, 18), (8192, 4, 16, 6, 5, 31)]
# (n, L, ell, B, levels)
FOLD = [(2048, 1, 2, 40, 5), (2048, 3, 5, 24, 5), (4096, 2, 4, 20, 5), (8192, 4, 16, 6, 4)]


@pytest.mark.parametrize("n,L,ell,B,levels,count", EXPAND)
def test_expand_batch_equals_single_queries(n, L, ell, B, levels, count):
    p = g.pir_make_params(n, 8, count, 4, L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + L)
    keys, packed = residues(gen, (levels, ell, 2), p), residues(gen, (B, 2), p)
    ex = g.pir_expander_create(p, levels, ell, keys)
    try:
        batch = torch.empty(B, count, 2, L, n, dtype=torch.int32, device="cuda")
        one = torch.empty(1, count, 2, L, n, dtype=torch.int32, device="cuda")
        g.pir_expand(ex, packed, B, count, batch)
        for b in (0, B // 2, B - 1):
            g.pir_expand(ex, packed[b:b + 1].contiguous(), 1, count, one)
            assert torch.equal(one[0], batch[b])
    finally:
        g.pir_expander_free(ex)


@pytest.mark.parametrize("n,L,ell,B,levels", FOLD)
def test_fold_batch_equals_single_queries(n, L, ell, B, levels):
    p = g.pir_make_params(n, 8, 1, 1 << levels, L)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + L)
    cts, rgsw = residues(gen, (B, 1 << levels, 2), p), residues(gen, (B, levels, 2 * ell, 2), p)
    batch = torch.empty(B, 2, L, n, dtype=torch.int32, device="cuda")
    one = torch.empty(1, 2, L, n, dtype=torch.int32, device="cuda")
    g.pir_fold(p, cts, B, levels, ell, rgsw, batch)
    for b in (0, B // 2, B - 1):
        g.pir_fold(p, cts[b:b + 1].contiguous(), 1, levels, ell, rgsw[b:b + 1].contiguous(), one)
        assert torch.equal(one[0], batch[b])
