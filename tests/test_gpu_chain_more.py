"""Kernels that start while their predecessor drains, on the GPU: the expansion and folding
chains, captured graphs, and scratch that moves between streams.  The same calls, alone and
synchronized, give what is expected; whole numbers: equal."""
import pytest

pytest.importorskip("torch")
import torch

import paper_2606_11536_gb300 as g

pytestmark = pytest.mark.gpu


def residues(p, lead, gen):
    x = torch.empty(*lead, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, q in enumerate(p.qs):
        x[..., j, :] = torch.randint(0, q, (*lead, p.n), generator=gen, dtype=torch.int32, device="cuda")
    return x


def database(n, D1, D2, L, gen, layout=0):
    p = g.pir_make_params(n, 8, D1, D2, L)
    raw = torch.randint(0, 256, (D1 * D2 * n,), generator=gen, dtype=torch.uint8, device="cuda")
    return p, g.pir_setup_db(p, raw, layout)


@pytest.fixture
def gen():
    gen = torch.Generator(device="cuda")
    gen.manual_seed(17)
    return gen


def test_expansion_and_folding_on_two_streams(gen):
    """Packed and folded answers in turn on two streams, their buffers rewritten in between: the
    scratch of one call is the next one's, on the same stream and on the other."""
    D1, D2, B, ell = 24, 8, 2, 4
    p, db = database(2048, D1, D2, 2, gen)
    ex = g.pir_expander_create(p, 5, ell, residues(p, (5, ell, 2), gen))
    try:
        packed = [residues(p, (B, 2), gen) for _ in range(3)]
        queries = [residues(p, (B, D1, 2), gen) for _ in range(3)]
        rgsw = [residues(p, (B, 3, 2 * ell, 2), gen) for _ in range(3)]

        def answer(k, q, w, out, stream=None):
            if k % 2:
                g.pir_answer_packed(db, ex, q, B, out, stream=stream)
            else:
                g.pir_answer_folded(db, q, B, ell, w, out, stream=stream)

        shapes = [(B, 2, 2, 2048), (B, D2, 2, 2, 2048)]
        alone = {}
        for k in (0, 1):
            for i in range(3):
                out = torch.empty(shapes[k], dtype=torch.int32, device="cuda")
                answer(k, (queries, packed)[k][i], rgsw[i], out)
                torch.cuda.synchronize()
                alone[k, i] = out
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        bufs = [[torch.empty_like(queries[0]), torch.empty_like(packed[0]), torch.empty_like(rgsw[0])] for _ in streams]
        outs = [[torch.empty(s, dtype=torch.int32, device="cuda") for s in shapes] for _ in streams]
        torch.cuda.synchronize()
        got = []
        for r in range(30):
            for t, s in enumerate(streams):
                k, i = (r + t) % 2, (r + t) % 3
                with torch.cuda.stream(s):
                    bufs[t][k].copy_((queries, packed)[k][i])
                    bufs[t][2].copy_(rgsw[i])
                    answer(k, bufs[t][k], bufs[t][2], outs[t][k], stream=s)
                    got.append((k, i, outs[t][k].clone()))
        torch.cuda.synchronize()
        for k, i, x in got:
            assert torch.equal(x, alone[k, i]), (k, i)
    finally:
        g.pir_expander_free(ex)
        g.pir_free_db(db)


@pytest.mark.parametrize("n,D1,D2,B,L", [(2048, 16, 16, 1, 2), (4096, 40, 12, 3, 3), (2048, 320, 64, 4, 2)])
def test_captured_answers_between_other_kernels(gen, n, D1, D2, B, L):
    """One graph, replayed with its query buffer rewritten before and its responses read after
    each replay on the same stream, and answers without a graph in between."""
    p, db = database(n, D1, D2, L, gen)
    try:
        qs = [residues(p, (B, D1, 2), gen) for _ in range(3)]
        alone = []
        for q in qs:
            r = torch.empty(B, D2, 2, L, n, dtype=torch.int32, device="cuda")
            g.pir_answer(db, q, B, r)
            torch.cuda.synchronize()
            alone.append(r)
        q, r, r2 = torch.empty_like(qs[0]), torch.empty_like(alone[0]), torch.empty_like(alone[0])
        torch.cuda.synchronize()
        graph = g.pir_graph_create(db, q, B, r)
        try:
            for k in range(30):
                q.copy_(qs[k % 3])
                g.pir_graph_launch(graph)
                got = r.clone()
                q.copy_(qs[(k + 1) % 3])
                g.pir_answer(db, q, B, r2)
                assert torch.equal(got, alone[k % 3]) and torch.equal(r2, alone[(k + 1) % 3]), k
        finally:
            g.pir_graph_destroy(graph)
    finally:
        g.pir_free_db(db)


def test_more_rows_than_there_can_be_are_refused():
    """Counts past 2^31 rows of 8 KiB and more: an error from the host, with nothing launched."""
    import ctypes as C

    p = g.pir_make_params(2048, 8, 1, 1, 1)
    x = torch.zeros(2048, dtype=torch.int32, device="cuda")
    for count in (1 << 31, 1 << 40, (1 << 63) + 1, (1 << 64) - 1):
        for f in (g.binding.lib().ntt_fwd, g.binding.lib().ntt_inv):
            assert f(C.byref(p), C.c_void_p(x.data_ptr()), count, None) == 4
    g.ntt_inv(p, g.ntt_fwd(p, x))
