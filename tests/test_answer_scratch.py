"""Device scratch that the server sets aside for a batch (host arithmetic), against what the answer
takes on the device."""
import types

import pytest

import paper_2606_11536_gb300 as g
from paper_2606_11536_gb300 import binding
from paper_2606_11536_gb300.serving import Request
from test_serving_host import make

PLAIN, LIMB, TENSOR = g.PIR_LAYOUT_PLAIN, g.PIR_LAYOUT_LIMB, g.PIR_LAYOUT_TENSOR


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2606_11536_gb300 import build
    build.build()


def params(n, L, D1, D2):
    return types.SimpleNamespace(n=n, L=L, D1=D1, D2=D2, log2p=8)


def test_small_batches_keep_both_copies():
    """Below 4096 rows the queries are transformed first: their 4 bytes per residue and the digits'
    8, of 2B rows padded to 4 and D1 padded to 64."""
    slots, ct = 2 * 4096, 2 * 2 * 4096 * 4
    for layout, D1 in ((PLAIN, 200), (LIMB, 224)):
        need = 3 * D1 * ct + slots * 256 * 8 * 8 + 3 * 20 * ct
        assert need > 3 * (2 * D1 + 20) * ct
        assert binding.answer_scratch_bytes(params(4096, 2, D1, 20), layout, 3) == need
    # one padded row of digits more than the copies that the queries no longer need
    p = params(4096, 2, 512, 20)
    assert binding.answer_scratch_bytes(p, PLAIN, 3) == max(3 * (2 * 512 + 20) * ct, slots * 512 * 8 * 8 + 3 * 20 * ct)
    # one query on the tensor layout: eight rows of digits
    p = params(4096, 2, 64, 32)
    assert binding.answer_scratch_bytes(p, TENSOR, 1) == 64 * ct + slots * 64 * 8 * 8 + 32 * ct


def test_server_counts_what_a_batch_takes():
    p = params(4096, 2, 200, 20)
    size = {nb: nb * 8 * 2 * 4096 * 220 + binding.answer_scratch_bytes(p, PLAIN, nb) for nb in range(1, 9)}
    assert size[4] > 4 * size[1]  # counted by the single query, a batch would take more than it was given
    clock, be, srv = make(streams=2, max_batch=8, scratch_budget=4 * size[1])
    srv.admit("a", p, None, layout=PLAIN)
    for k in range(6):
        srv.submit(Request(k, "a", k, 0.0))
    left, want = 4 * size[1], []
    for waiting in (6, 6 - max(nb for nb in size if nb <= 6 and size[nb] <= left)):  # two streams
        fits = [nb for nb in size if nb <= waiting and size[nb] <= left]
        want += [max(fits)] if fits else []
        left -= size[want[-1]] if fits else 0
    srv.poll()
    assert [len(q) for _, q in be.batches] == want and sum(want) < 4 and srv.scratch_in_flight == 4 * size[1] - left
    for t in range(1, 6):
        clock.t = float(t)
        srv.poll()
    assert srv.pending() == 0 and srv.scratch_in_flight == 0 and len(srv.done) == 6


@pytest.mark.gpu
@pytest.mark.parametrize("layout,n,L,D1,D2,B", [
    (PLAIN, 4096, 2, 512, 64, 1), (PLAIN, 8192, 2, 200, 20, 2), (PLAIN, 8192, 3, 130, 64, 3), (PLAIN, 4096, 2, 384, 64, 31),
    (PLAIN, 4096, 2, 1024, 16, 33), (LIMB, 8192, 2, 96, 20, 1), (LIMB, 4096, 3, 160, 32, 5), (LIMB, 4096, 2, 512, 32, 32),
    (TENSOR, 8192, 2, 128, 32, 1), (TENSOR, 4096, 2, 512, 64, 17),
])
def test_an_answer_takes_no_more(layout, n, L, D1, D2, B):
    import torch

    p = g.pir_make_params(n, 8, D1, D2, L)
    db = g.pir_setup_db(p, torch.zeros(D1 * D2 * n, dtype=torch.uint8, device="cuda"), layout)
    try:
        q = torch.zeros(B * D1 * 2 * L * n, dtype=torch.int32, device="cuda")
        r = torch.empty(B * D2 * 2 * L * n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        g.pir_release_memory()
        before = torch.cuda.mem_get_info()[0]
        g.pir_answer(db, q, B, r)
        torch.cuda.synchronize()
        taken = before - torch.cuda.mem_get_info()[0]
        g.pir_release_memory()
        assert taken <= binding.answer_scratch_bytes(p, layout, B) + (64 << 20), taken  # the pool grows in steps
    finally:
        g.pir_free_db(db)
