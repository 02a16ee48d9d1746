"""Short pieces of a long answer on the plain layout: each takes the path of its own size, on the
tensor cores or not, and all add up."""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu


def instance(n, L, D1, D2, B, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    p = g.pir_make_params(n, 8, D1, D2, L)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    q = torch.empty(B, D1, 2, L, n, dtype=torch.int32, device="cuda")
    for j, m in enumerate(p.qs):
        q[..., j, :] = torch.randint(0, m, (B, D1, 2, n), generator=gen, dtype=torch.int32, device="cuda")
    return g.pir_setup_db(p, raw), q


def streamed(db, q, B, pieces, r, tile=0):
    s = g.pir_answer_begin(db, B, max(pieces), tile=tile)
    i0 = 0
    for kc in pieces:
        g.pir_answer_chunk(s, q[:, i0:i0 + kc].contiguous(), i0, kc)
        i0 += kc
    g.pir_answer_end(s, r)


@pytest.mark.parametrize("n,L,D2,B,pieces", [
    (2048, 2, 132, 3, (130, 1, 63, 64, 65)),         # a long one first, then every side of a 64-row block
    (2048, 1, 512, 8, (16, 200, 128, 127, 191, 192)),
    (4096, 2, 20, 16, (7, 150, 50)),
    (2048, 3, 64, 33, (40, 300, 20)),
    (2048, 1, 516, 2, (129, 100, 3)),                # wider than the scans
])
def test_mixed_pieces_equal_the_integer_tiles(n, L, D2, B, pieces):
    D1 = sum(pieces)
    db, q = instance(n, L, D1, D2, B, seed=D1)
    try:
        want, r = (torch.empty(B, D2, 2, L, n, dtype=torch.int32, device="cuda") for _ in range(2))
        g.pir_answer_ex(db, q, B, want, tile=6)
        streamed(db, q, B, pieces, r)
        assert torch.equal(r, want)
        for k_chunk in (max(pieces), 130, 17):  # ends in a short chunk
            r.zero_()
            g.pir_answer_ex(db, q, B, r, k_chunk=k_chunk)
            assert torch.equal(r, want), k_chunk
        g.pir_check_device()
    finally:
        g.pir_free_db(db)


@pytest.mark.parametrize("D2,B,piece,tile", [(512, 4, 16, 8), (128, 16, 16, 5), (256, 2, 8, 7)])
def test_short_pieces_of_a_session_take_their_own_path(D2, B, piece, tile):
    """Pieces of 16 rows ran on the digit GEMM whenever the session allowed for 128 and more: 26.2
    against 4.8 ms here (512 columns, 4 queries)."""
    n, L, D1 = 4096, 2, 512
    db, q = instance(n, L, D1, D2, B, seed=1)
    try:
        r = torch.empty(B, D2, 2, L, n, dtype=torch.int32, device="cuda")
        part = q[:, :piece].contiguous()

        def ms(tile):
            best = 1e9
            for _ in range(4):
                s = g.pir_answer_begin(db, B, D1, tile=tile)
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                for i0 in range(0, D1, piece):
                    g.pir_answer_chunk(s, part, i0, piece)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
                g.pir_answer_end(s, r)
            return best

        assert ms(0) <= 1.5 * ms(tile)
    finally:
        g.pir_free_db(db)
