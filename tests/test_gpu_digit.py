"""The tensor-core GEMM over in-kernel digits (tile 9 of the plain layout, 4 of the limb
layout): equal, word for word, to the CUDA-core and INT8 tiles and to the oracle at the
edges of its tiles (64-row blocks, 1024- and 512-row sums, 32-column tiles, accumulator
widths from 16 to 256 columns)."""
import numpy as np
import pytest

import paper_2606_11536_gb300 as g
import synth
from gpu_util import empty_u32, from_dev, random_queries, to_dev

pytestmark = pytest.mark.gpu

DIGIT = 9


def device_db(p, seed, layout=0):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nbytes = p.D1 * p.D2 * p.n * p.log2p // 8
    raw = torch.randint(0, 256, (nbytes,), generator=gen, dtype=torch.uint8, device="cuda")
    return g.pir_setup_db(p, raw, layout)


def device_queries(p, B, seed):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    q = torch.empty(B, p.D1, 2, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, prime in enumerate(p.qs):
        q[..., j, :] = torch.randint(0, prime, (B, p.D1, 2, p.n), generator=gen, dtype=torch.int32, device="cuda")
    return q


def answer(db, q, B, **kw):
    p = db.params
    r = empty_u32(B * p.D2 * 2 * p.L * p.n)
    g.pir_answer_ex(db, q, B, r, **kw)
    g.pir_check_device()
    return r


@pytest.mark.parametrize("D1,D2,L,batches", [
    (63, 4, 2, (2, 3)),            # less than one block of rows, one quad of columns
    (65, 28, 1, (2, 12, 17)),      # one row into a second block
    (129, 36, 2, (3, 16, 24, 25)),  # two column tiles; 192 and 200 accumulator columns
    (192, 132, 3, (2, 5, 31, 32)),  # ragged columns over three primes
    (1025, 68, 1, (4, 33)),        # one row into a second 1024-row sum; 256 + 8 rows
    (2100, 32, 1, (9, 48, 65)),    # three sums; two and three tiles of query rows
])
def test_equals_the_cuda_core_tiles(D1, D2, L, batches):
    import torch
    p = g.pir_make_params(2048, 8, D1, D2, L)
    db = device_db(p, D1)
    try:
        for B in batches:
            q = device_queries(p, B, B)
            ref = answer(db, q, B, tile=5)
            assert torch.equal(answer(db, q, B, tile=DIGIT), ref), B
            assert torch.equal(answer(db, q, B, tile=DIGIT, k_chunk=100), ref), B  # accumulated chunks
            assert torch.equal(answer(db, q, B), ref), B
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("D1,D2,L,batches", [
    (32, 4, 2, (1, 2)),             # half a block of rows, one query
    (96, 28, 1, (3, 12, 17)),       # a block and a half
    (160, 36, 2, (1, 16, 24, 25)),  # two column tiles; 192 and 200 accumulator columns
    (544, 68, 1, (4, 33)),          # 32 rows into a second 512-row sum; 256 + 8 rows
    (1600, 32, 1, (1, 48, 65)),     # four sums; two and three tiles of query rows
])
def test_limb_layout_equals_the_int8_tiles(D1, D2, L, batches):
    import torch
    p = g.pir_make_params(2048, 8, D1, D2, L)
    db = device_db(p, D1, layout=1)
    try:
        for B in batches:
            q = device_queries(p, B, B)
            ref = answer(db, q, B, tile=1)
            assert torch.equal(answer(db, q, B, tile=4), ref), B
            assert torch.equal(answer(db, q, B, tile=4, k_chunk=96), ref), B  # accumulated chunks
            assert torch.equal(answer(db, q, B), ref), B
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("layout,tile", [(0, DIGIT), (1, 4)])
def test_extreme_residues_and_the_oracle(orc, layout, tile):
    """Queries of q - 1 everywhere (the largest digits of every prime) and uniform ones."""
    n, D1, D2, L, B = 2048, 160, 40, 2, 3
    p, P = g.pir_make_params(n, 16, D1, D2, L), orc.make_params(n, 16, D1, D2, L)
    raw = synth.raw_db(5, synth.raw_db_bytes(n, 16, D1, D2))
    db = g.pir_setup_db(p, raw, layout)
    try:
        Q = random_queries(P, B, 6)
        Q[1] = np.array(P.qs, dtype=np.uint32)[None, None, :, None] - 1
        R = from_dev(answer(db, to_dev(Q), B, tile=tile), (B, D2, 2, L, n))
        assert np.array_equal(R, orc.answer(P, raw, Q))
    finally:
        g.pir_free_db(db)


def test_sums_at_the_f32_bound():
    """Digit pairs of -128 times -128 over whole 1024-row sums: exactly 2^24."""
    import torch
    D1, D2, B, v = 1024, 32, 2, 0x7F7F80  # digits -128, -128, -128, 1
    p = g.pir_make_params(2048, 23, D1, D2, 1)
    coeff = np.zeros(p.n, dtype=np.uint32)
    coeff[0] = v  # a constant polynomial is the same residue in every slot
    bits = np.unpackbits(coeff.view(np.uint8).reshape(-1, 4), axis=1, bitorder="little")[:, :23]
    poly = torch.from_numpy(np.packbits(bits.reshape(-1), bitorder="little")).cuda()
    db = g.pir_setup_db(p, poly.repeat(D1 * D2))
    try:
        q = torch.zeros(B, D1, 2, 1, p.n, dtype=torch.int32, device="cuda")
        q[..., 0] = v
        r = answer(db, q, B, tile=DIGIT).cpu().numpy().view(np.uint32).reshape(B, D2, 2, p.n)
        want = np.zeros(p.n, dtype=np.uint32)
        want[0] = D1 * v * v % p.qs[0]
        assert np.array_equal(r, np.broadcast_to(want, r.shape))
    finally:
        g.pir_free_db(db)


def test_one_query_is_refused():
    p = g.pir_make_params(2048, 8, 64, 8, 1)
    db = device_db(p, 1)
    try:
        with pytest.raises(g.PirError):
            answer(db, device_queries(p, 1, 1), 1, tile=DIGIT)
    finally:
        g.pir_free_db(db)
