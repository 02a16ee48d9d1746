"""The device scratch of batched answers: no copy of the queries that nothing reads, the smaller
form where memory is short, and pieces inside a chunk."""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu
GIB = 1 << 30


def instance(n, L, D1, D2, B, layout=0, seed=1):
    """(database, queries) of random records and residues."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    p = g.pir_make_params(n, 8, D1, D2, L)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    q = torch.empty(B, D1, 2, L, n, dtype=torch.int32, device="cuda")
    for j, m in enumerate(p.qs):
        q[..., j, :] = torch.randint(0, m, (B, D1, 2, n), generator=gen, dtype=torch.int32, device="cuda")
    return g.pir_setup_db(p, raw, layout), q


def responses(db, B):
    p = db.params
    return torch.empty(B, p.D2, 2, p.L, p.n, dtype=torch.int32, device="cuda")


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def give_back():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    g.pir_release_memory()


@pytest.mark.parametrize("layout", [g.PIR_LAYOUT_PLAIN, g.PIR_LAYOUT_LIMB, g.PIR_LAYOUT_TENSOR])
def test_no_copy_that_nothing_reads(layout):
    """32 queries of 256 ciphertexts, transformed straight into the digits: 1 GiB of digits (8 bytes
    a residue, 2B rows) and 32 MiB of results (D2 = 32 of 64 rows), not another 512 MiB."""
    n, L, D1, D2, B = 4096, 2, 256, 32, 32
    db, q = instance(n, L, D1, D2, B, layout)
    try:
        r = responses(db, B)
        give_back()
        before = free()
        g.pir_answer(db, q, B, r)
        taken = before - free()
        need = L * n * 2 * B * (8 * D1 + 4 * D2)
        assert GIB <= need and taken <= need + (128 << 20), (taken, need)  # the pool grows in steps
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("layout", [g.PIR_LAYOUT_PLAIN, g.PIR_LAYOUT_LIMB])
@pytest.mark.parametrize("how", ["answer", "session"])
def test_smaller_pieces_where_memory_is_short(layout, how):
    """The digits of 32 queries of 256 ciphertexts are 1 GiB, in the smaller form 512 MiB: with
    about 800 MiB left (and a session's 512 MiB of transformed queries) only the latter fits."""
    n, L, D1, D2, B = 4096, 2, 256, 8, 32
    db, q = instance(n, L, D1, D2, B, layout, seed=3)
    filler = None
    try:
        want, r = responses(db, B), responses(db, B)
        g.pir_answer(db, q, B, want)
        left = (800 << 20) + (512 << 20) * (how == "session")
        give_back()
        filler = torch.empty(free() - left, dtype=torch.uint8, device="cuda")
        before = free()
        assert before < left + (64 << 20)
        if how == "answer":
            g.pir_answer(db, q, B, r)
        else:
            s = g.pir_answer_begin(db, B, D1)
            g.pir_answer_chunk(s, q, 0, D1)
            g.pir_answer_end(s, r)
        torch.cuda.synchronize()
        assert torch.equal(r, want)
        g.pir_check_device()
    finally:
        filler = None
        give_back()
        g.pir_free_db(db)


@pytest.mark.parametrize("layout,tile", [(g.PIR_LAYOUT_PLAIN, 6), (g.PIR_LAYOUT_LIMB, 3)])
def test_pieces_of_a_chunk_from_transformed_queries(layout, tile):
    """More than 1 GiB of digits are made and multiplied in pieces, here of 1088 rows of 2176 (a
    session transforms its queries first); against the integer tiles."""
    n, L, D1, D2, B = 2048, 1, 2176, 4, 32
    db, q = instance(n, L, D1, D2, B, layout, seed=5)
    try:
        want, r = responses(db, B), responses(db, B)
        g.pir_answer_ex(db, q, B, want, tile=tile)
        g.pir_answer(db, q, B, r)
        assert torch.equal(r, want)
        r.zero_()
        s = g.pir_answer_begin(db, B, D1)
        g.pir_answer_chunk(s, q, 0, D1)
        g.pir_answer_end(s, r)
        assert torch.equal(r, want)
        g.pir_check_device()
    finally:
        give_back()
        g.pir_free_db(db)
