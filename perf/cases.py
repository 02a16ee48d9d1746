"""What a server built on this library has it do, as cases that can be timed.

The cases go through the package's public calls on the shapes of the repository's own
configurations, tests and benchmark, and on ragged ones between them:

  answer   the first-dimension answer to a batch of queries on a resident database
           (plain, limb or tensor layout; a direct call or a captured graph)
  packed   one packed ciphertext per query, expanded and answered (host buffers: the
           queries come off the network and the responses go back to it)
  folded   the answer folded over the remaining dimensions to one ciphertext
  ntt      the standalone transforms, in place
  lwe      the scalar-HE database product

Ciphertexts, keys and database bytes are uniform, as encrypted data and encoded
records are.
"""
import math

import numpy as np
import torch

import paper_2606_11536_gb300 as g

LAYOUTS = {"plain": g.PIR_LAYOUT_PLAIN, "limb": g.PIR_LAYOUT_LIMB, "tensor": g.PIR_LAYOUT_TENSOR}

# The largest listed answer: 8 GiB of records, 32 GiB resident, 32 queries.
MOST_MACS = 8192 * 2048 * 512 * 64
MOST_RESIDENT = 8 << 30  # drawn databases stay quick to make


def answer(name, n, log2p, D1, D2, B, layout="plain", L=2, modswitch=False, via="call"):
    return dict(name=name, kind="answer", layout=layout, n=n, L=L, log2p=log2p, D1=D1, D2=D2, B=B,
                modswitch=modswitch, via=via)


def listed():
    return [
        # the smallest configuration: one query on a 768 KiB database, bound by latency and launches
        answer("answer_tiny_b1", 2048, 12, 16, 16, 1),
        # one query on a 1 GiB database: the scan streams 4 GiB
        answer("answer_1g_b1", 4096, 16, 512, 256, 1),
        # a few queries on an odd-shaped database over three primes
        answer("answer_ragged_b3", 4096, 12, 301, 132, 3, L=3),
        # a small batch at the small ring, served from a captured graph, responses over one prime
        answer("answer_1g_n2048_b8", 2048, 16, 512, 512, 8, modswitch=True, via="graph"),
        # the largest: a full batch on an 8 GiB database
        answer("answer_8g_b32", 4096, 16, 2048, 512, 32),
        # the layout the server keeps its databases in, at its batch cap
        answer("tensor_1g_b32", 4096, 16, 512, 256, 32, layout="tensor"),
        # the byte-limb layout
        answer("limb_512m_b32", 2048, 16, 512, 256, 32, layout="limb"),
        # encoding-sized transforms: 2 GiB of polynomials, forward
        dict(name="ntt_fwd_n4096", kind="ntt", forward=True, n=4096, L=2, count=65536),
        # inverse transforms of an odd number of polynomials at the large ring, three primes
        dict(name="ntt_inv_n8192", kind="ntt", forward=False, n=8192, L=3, count=1001),
        # a few clients' packed queries, host to host, responses over one prime
        dict(name="packed_1g_b4", kind="packed", n=4096, L=2, log2p=16, D1=512, D2=256, B=4, ell=4, modswitch=True),
        # a few queries folded to one ciphertext each
        dict(name="folded_1g_b4", kind="folded", n=4096, L=2, log2p=16, D1=512, D2=256, B=4, ell=4),
        # the scalar-HE product: a 1 GiB INT8 database, a full batch
        dict(name="lwe_1g_b32", kind="lwe", D1=32768, D0=32768, B=32),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["answer"] * 6 + ["tensor", "tensor", "limb", "ntt", "ntt", "packed", "folded", "lwe", "lwe"])
    n, L = rng.choice([2048, 4096, 4096, 8192]), rng.choice([1, 2, 2, 2, 3, 4])
    if kind == "ntt":
        return dict(kind="ntt", forward=rng.random() < 0.5, n=n, L=L, count=_log(rng, 1, 65536 * 4096 * 2 // (n * L)))
    if kind == "lwe":
        return dict(kind="lwe", D1=_log(rng, 200, 32768), D0=16 * _log(rng, 16, 2048), B=_log(rng, 1, 48))
    if kind == "packed":
        return dict(kind="packed", n=4096, L=rng.choice([2, 3]), log2p=rng.choice([8, 16]), D1=_log(rng, 16, 512),
                    D2=4 * _log(rng, 4, 64), B=_log(rng, 1, 16), ell=rng.choice([4, 5, 6]), modswitch=rng.random() < 0.5)
    if kind == "folded":
        return dict(kind="folded", n=rng.choice([2048, 4096]), L=rng.choice([2, 3]), log2p=rng.choice([8, 16]),
                    D1=_log(rng, 16, 512), D2=2 ** rng.randint(3, 8), B=_log(rng, 1, 16), ell=rng.choice([4, 5, 6]))
    layout = "plain" if kind == "answer" else kind
    rows, cols = {"plain": (1, 4), "limb": (32, 4), "tensor": (64, 32)}[layout]
    while True:
        D1 = rows * _log(rng, max(1, 16 // rows), 2048 // rows)
        D2 = cols * _log(rng, max(1, 16 // cols), 512 // cols)
        B = _log(rng, 1, 64)
        per = 8 if layout == "tensor" else 4
        if n * L * D1 * D2 * per <= MOST_RESIDENT and n * L * D1 * D2 * 2 * B <= MOST_MACS // 4:
            return dict(kind="answer", layout=layout, n=n, L=L, log2p=rng.choice([8, 12, 16]), D1=D1, D2=D2, B=B,
                        modswitch=rng.random() < 0.3, via=rng.choice(["call", "call", "graph"]))


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _residues(gen, lead, p):
    """Uniform canonical residues [*lead][L][n]."""
    out = torch.empty(*lead, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, q in enumerate(p.qs):
        out[..., j, :] = torch.randint(0, q, (*lead, p.n), generator=gen, dtype=torch.int32, device="cuda")
    return out


def _raw(gen, nbytes):
    words = torch.randint(-2**31, 2**31 - 1, ((nbytes + 3) // 4,), generator=gen, dtype=torch.int32, device="cuda")
    return words.view(torch.uint8)[:nbytes]


class State:
    """What a server holds between calls: handles and buffers; the handles go back with it."""

    def __init__(self, case):
        self.case = case
        self.db = self.graph = self.expander = None

    def __del__(self):
        if self.graph is not None:
            g.pir_graph_destroy(self.graph)
        if self.expander is not None:
            g.pir_expander_free(self.expander)
        if self.db is not None:
            g.pir_free_db(self.db)


def _sizes(case):
    """(database bytes, levels of expansion, levels of folding)"""
    raw = case["D1"] * case["D2"] * case["n"] * case["log2p"] // 8
    return raw, max(0, (case["D1"] - 1).bit_length()), max(0, (case["D2"] - 1).bit_length())


def _inputs(case, seed):
    """The tensors of a case, made from the seed alone: (params, raw database, the others by name)."""
    gen, kind = _generator(seed), case["kind"]
    if kind == "lwe":
        db = _raw(gen, case["D1"] * case["D0"]).view(torch.int8)
        q = _raw(gen, 4 * case["B"] * case["D0"]).view(torch.int32)
        return None, db, {"queries": q}
    if kind == "ntt":
        p = g.pir_make_params(case["n"], 16, 1, 1, case["L"])
        return p, None, {"polys": _residues(gen, (case["count"],), p)}
    p = g.pir_make_params(case["n"], case["log2p"], case["D1"], case["D2"], case["L"])
    nraw, up, down = _sizes(case)
    raw, B = _raw(gen, nraw), case["B"]
    if kind == "packed":
        return p, raw, {"keys": _residues(gen, (up, case["ell"], 2), p), "queries": _residues(gen, (B, 2), p)}
    t = {"queries": _residues(gen, (B, case["D1"], 2), p)}
    if kind == "folded":
        t["rgsw"] = _residues(gen, (B, down, 2 * case["ell"], 2), p)
    return p, raw, t


def prepare(case, seed):
    s = State(case)
    p, raw, t = _inputs(case, seed)
    kind = case["kind"]
    s.p, s.t = p, t
    if kind == "lwe":
        s.raw = raw
        s.out = torch.empty(case["B"], case["D1"], dtype=torch.int32, device="cuda")
        return s
    if kind == "ntt":
        return s
    s.db = g.pir_setup_db(p, raw, LAYOUTS[case.get("layout", "plain")])
    del raw
    torch.cuda.empty_cache()  # the record bytes are no longer needed beside the resident form
    B = case["B"]
    s.flags = g.PIR_ANSWER_MODSWITCH if case.get("modswitch") else 0
    rows = (p.n,) if s.flags else (p.L, p.n)
    if kind == "packed":
        s.expander = g.pir_expander_create(p, _sizes(case)[1], case["ell"], t["keys"])
        s.host_in = t["queries"].cpu().pin_memory()
        s.out = torch.empty(B, case["D2"], 2, *rows, dtype=torch.int32, pin_memory=True)
    elif kind == "folded":
        s.out = torch.empty(B, 2, *rows, dtype=torch.int32, device="cuda")
    else:
        s.out = torch.empty(B, case["D2"], 2, *rows, dtype=torch.int32, device="cuda")
        if case["via"] == "graph":
            s.graph = g.pir_graph_create(s.db, t["queries"], B, s.out, flags=s.flags)
    return s


def run(s):
    c, t = s.case, s.t
    kind = c["kind"]
    if kind == "ntt":
        return (g.ntt_fwd if c["forward"] else g.ntt_inv)(s.p, t["polys"])
    if kind == "lwe":
        return g.pir_lwe_answer(s.raw, c["D1"], c["D0"], t["queries"], c["B"], s.out)
    if kind == "packed":
        return g.pir_answer_packed(s.db, s.expander, s.host_in, c["B"], s.out, flags=s.flags)
    if kind == "folded":
        return g.pir_answer_folded(s.db, t["queries"], c["B"], c["ell"], t["rgsw"], s.out)
    if s.graph is not None:
        g.pir_graph_launch(s.graph)
        return s.out
    if s.flags:
        return g.pir_answer_ex(s.db, t["queries"], c["B"], s.out, flags=s.flags)
    return g.pir_answer(s.db, t["queries"], c["B"], s.out)


def work(case):
    """Bytes: inputs read once (the database in its resident form), outputs written once.
    Operations: a multiply and an add per modular product, and per butterfly."""
    kind = case["kind"]
    if kind == "lwe":
        D1, D0, B = case["D1"], case["D0"], case["B"]
        return {"bytes": D1 * D0 + 4 * B * (D0 + D1), "flops": 2 * D1 * D0 * B}
    n, L = case["n"], case["L"]
    butterflies = n // 2 * int(math.log2(n))  # of one row
    if kind == "ntt":
        rows = case["count"] * L
        return {"bytes": 8 * rows * n, "flops": 2 * rows * butterflies}
    D1, D2, B = case["D1"], case["D2"], case["B"]
    ct = 2 * L * n * 4
    _, up, down = _sizes(case)
    db = L * n * D1 * D2 * (8 if case.get("layout") == "tensor" else 4)
    macs = L * n * D1 * D2 * 2 * B
    resp = ct // L if case.get("modswitch") else ct
    if kind == "packed":
        ell, cts = case["ell"], 2 ** up - 1  # key switches of one query's expansion
        rows = B * (2 * L + cts * (L + ell * L) + D2 * 2 * L)
        macs += B * cts * 2 * ell * L * n
        return {"bytes": db + B * ct + up * ell * ct + B * D2 * resp, "flops": 2 * (macs + rows * butterflies)}
    if kind == "folded":
        ell, pairs = case["ell"], D2 - 1
        rows = B * (D1 * 2 * L + down * 2 * ell * 2 * L + pairs * (2 * L + 2 * ell * L) + 2 * L)
        macs += B * pairs * 2 * ell * 2 * L * n
        return {"bytes": db + B * D1 * ct + B * down * 2 * ell * ct + B * ct, "flops": 2 * (macs + rows * butterflies)}
    rows = B * (D1 + D2) * 2 * L
    return {"bytes": db + B * D1 * ct + B * D2 * resp, "flops": 2 * (macs + rows * butterflies)}


# --- the same results from the definitions, in 64-bit integers -----------------------


def _roots(n, q):
    """psi^brv(i) and its inverse, for the smallest generator base whose psi has order 2n."""
    h = 2
    while pow(pow(h, (q - 1) // (2 * n), q), n, q) != q - 1:
        h += 1
    psi, bits = pow(h, (q - 1) // (2 * n), q), n.bit_length() - 1
    brv = [int(format(i, "0%db" % bits)[::-1], 2) for i in range(n)]
    tables = []
    for w in (psi, pow(psi, -1, q)):
        powers = [1] * n
        for i in range(1, n):
            powers[i] = powers[i - 1] * w % q
        tables.append(torch.tensor([powers[b] for b in brv], dtype=torch.int64, device="cuda"))
    return tables


def _ntt(a, q, table):
    """Forward negacyclic transform of int64 rows [..., n]."""
    n, m = a.shape[-1], 1
    while m < n:
        v = a.reshape(*a.shape[:-1], m, 2, n // (2 * m))
        x, y = v[..., 0, :], v[..., 1, :] * table[m:2 * m, None] % q
        a = torch.stack(((x + y) % q, (x - y) % q), dim=-2).reshape(a.shape)
        m *= 2
    return a


def _intt(a, q, table):
    n = a.shape[-1]
    m = n // 2
    while m >= 1:
        v = a.reshape(*a.shape[:-1], m, 2, n // (2 * m))
        x, y = v[..., 0, :], v[..., 1, :]
        a = torch.stack(((x + y) % q, (x - y) * table[m:2 * m, None] % q), dim=-2).reshape(a.shape)
        m //= 2
    return a * pow(n, -1, q) % q


def _coefficients(raw, log2p, n, count):
    """Plaintext polynomials [count][n] of the record bytes."""
    if log2p == 8:
        return raw.reshape(count, n).to(torch.int64)
    if log2p == 16:
        b = raw.reshape(count, n, 2).to(torch.int64)
        return b[..., 0] + 256 * b[..., 1]
    b = raw.reshape(count, n // 2, 3).to(torch.int64)  # two 12-bit coefficients in three bytes
    return torch.stack((b[..., 0] + 256 * (b[..., 1] & 15), (b[..., 1] >> 4) + 16 * b[..., 2]), dim=-1).reshape(count, n)


def _exact_answer(case, seed):
    p, raw, t = _inputs(case, seed)
    n, D1, D2, B = case["n"], case["D1"], case["D2"], case["B"]
    out = torch.empty(B, D2, 2, p.L, n, dtype=torch.int64, device="cuda")
    plain = _coefficients(raw, case["log2p"], n, D1 * D2).reshape(D1, D2, n)
    for j, q in enumerate(p.qs):
        fwd, inv = _roots(n, q)
        acc = torch.zeros(B, D2, 2, n, dtype=torch.int64, device="cuda")
        for i in range(D1):
            query = _ntt(t["queries"][:, i, :, j, :].to(torch.int64), q, fwd)  # [B][2][n]
            acc = (acc + query[:, None] * _ntt(plain[i], q, fwd)[None, :, None]) % q
        out[:, :, :, j] = _intt(acc, q, inv)
    return out.to(torch.int32)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ntt" and case["count"] * case["L"] * case["n"] <= 1 << 27:
        p, _, t = _inputs(case, seed)
        a = t["polys"].to(torch.int64)
        for j, q in enumerate(p.qs):
            fwd, inv = _roots(p.n, q)
            a[:, j] = _ntt(a[:, j], q, fwd) if case["forward"] else _intt(a[:, j], q, inv)
        return a.to(torch.int32)
    if kind == "lwe" and case["D1"] * case["D0"] <= 1 << 28:
        _, db, t = _inputs(case, seed)
        a = db.reshape(case["D1"], case["D0"]).to(torch.float64)
        q = t["queries"].reshape(case["B"], case["D0"]).to(torch.int64) & 0xFFFFFFFF
        lo, hi = (((q >> s) & 0xFFFF).to(torch.float64) for s in (0, 16))  # sums below 2^38: exact
        v = ((lo @ a.T).to(torch.int64) + ((hi @ a.T).to(torch.int64) << 16)) & 0xFFFFFFFF
        return torch.from_numpy(v.cpu().numpy().astype(np.uint32).view(np.int32))
    if kind == "answer" and not case["modswitch"]:
        residues = case["D1"] * case["D2"] * case["n"]
        if residues <= 1 << 28 and case["L"] * residues * case["B"] <= 1 << 31:
            return _exact_answer(case, seed)
    return None
