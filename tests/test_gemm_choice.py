"""The kernel that tile 0 stands for, as a tile id (host arithmetic, no GPU)."""
import pytest

import paper_2606_11536_gb300 as g

PLAIN, LIMB, TENSOR = g.PIR_LAYOUT_PLAIN, g.PIR_LAYOUT_LIMB, g.PIR_LAYOUT_TENSOR


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2606_11536_gb300 import build
    build.build()


@pytest.mark.parametrize("layout,D1,D2,B,tile", [
    (PLAIN, 512, 256, 1, 7), (PLAIN, 4096, 512, 1, 7),  # one query: the staged scan of long slots,
    (PLAIN, 16, 16, 1, 10), (PLAIN, 64, 512, 2, 10),    # the direct one of short or odd ones
    (PLAIN, 16, 16, 16, 10),                            # more than eight rows of short slots
    (PLAIN, 100, 1024, 1, 1),                           # too wide for the scans
    (PLAIN, 128, 16, 2, 9), (PLAIN, 4096, 512, 32, 9),  # the digit GEMM from 128 rows on,
    (PLAIN, 127, 16, 6, 9), (PLAIN, 64, 64, 4, 9),      # and below where its cost says so
    (LIMB, 32, 4, 1, 4), (TENSOR, 512, 256, 32, 5), (TENSOR, 64, 96, 1, 1), (TENSOR, 64, 128, 40, 1),
])
def test_choice(layout, D1, D2, B, tile):
    assert g.pir_gemm_choice(layout, D1, D2, B) == tile


def test_every_choice_is_a_tile():
    for layout in (PLAIN, LIMB, TENSOR):
        for D1 in (1, 16, 64, 127, 128, 1000):
            for D2 in (4, 32, 132, 256, 512, 516, 1024):
                for B in (1, 2, 3, 4, 5, 16, 33, 64):
                    assert 1 <= g.pir_gemm_choice(layout, D1, D2, B) <= g.pir_gemm_tiles(layout)


def test_arguments():
    for bad in ((3, 16, 16, 1), (PLAIN, 0, 16, 1), (PLAIN, 16, 0, 1), (PLAIN, 16, 16, 0)):
        with pytest.raises(g.PirError) as ei:
            g.pir_gemm_choice(*bad)
        assert ei.value.status == 1


@pytest.mark.gpu
@pytest.mark.parametrize("n,D1,D2,B", [(4096, 16, 16, 16), (2048, 16, 4, 40), (4096, 64, 16, 4)])
def test_autotune_reaches_the_built_in_choice(n, D1, D2, B):
    """Small databases with many queries, where tile 0 is the direct scan and 1.6 times as fast as
    the GEMM tiles (16 x 16, 16 queries, 80 against 128 us): the autotuner finds it.  Equal words."""
    import torch

    assert g.pir_gemm_choice(PLAIN, D1, D2, B) == 10
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    p = g.pir_make_params(n, 8, D1, D2, 2)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    db = g.pir_setup_db(p, raw)
    try:
        q = torch.randint(0, min(p.qs), (B, D1, 2, 2, n), generator=gen, dtype=torch.int32, device="cuda")
        r0, r1, r2 = (torch.empty(B, D2, 2, 2, n, dtype=torch.int32, device="cuda") for _ in range(3))
        best = g.pir_autotune(db, B)
        g.pir_answer(db, q, B, r0)
        g.pir_answer_ex(db, q, B, r1, **best)
        g.pir_answer_ex(db, q, B, r2, tile=10)
        assert torch.equal(r0, r1) and torch.equal(r0, r2)

        def ms(**opts):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            times = []
            for _ in range(30):
                a.record()
                g.pir_answer_ex(db, q, B, r1, **opts)
                b.record()
                b.synchronize()
                times.append(a.elapsed_time(b))
            return min(times)

        assert ms(**best) <= 1.4 * ms(), best
    finally:
        g.pir_free_db(db)
