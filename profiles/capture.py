"""The program behind the captures in this folder: three calls of one case, small enough that a
capture of many counters ends in seconds, with inputs larger than L2.

    python profiles/capture.py CASE && ncu --clock-control none ... python profiles/capture.py CASE
"""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import torch  # noqa: E402

import paper_2606_11536_gb300 as g  # noqa: E402

CASES = {
    # answers: layout, n, log2 p, D1, D2, queries, tile
    "digit": ("plain", 2048, 16, 512, 256, 32, 0), "limb": ("limb", 2048, 16, 512, 256, 32, 0),
    "tensor": ("tensor", 2048, 16, 512, 256, 32, 0), "tensor2": ("tensor", 2048, 16, 512, 256, 32, 2),
    "plain6": ("plain", 2048, 16, 512, 256, 32, 6), "limb3": ("limb", 2048, 16, 512, 256, 32, 3),
    "scan": ("plain", 4096, 16, 512, 256, 1, 0), "direct": ("plain", 4096, 8, 256, 64, 1, 0),
    # transforms in place: n, primes, polynomials
    "ntt4096": (4096, 2, 65536), "ntt8192": (8192, 3, 10000),
    # expansion to `count` ciphertexts: n, primes, levels, digits, queries
    "expand": (4096, 2, 9, 4, 4),
    # the scalar-HE product: rows, bytes a row, queries
    "lwe": (8192, 32768, 32), "dp4a": (32768, 32768, 1),
}


def words(*shape, lo=-2**31, hi=2**31 - 1, dtype=torch.int32):
    return torch.randint(lo, hi, shape, dtype=dtype, device="cuda")


def residues(p, *lead):
    x = torch.empty(*lead, p.L, p.n, dtype=torch.int32, device="cuda")
    for j, q in enumerate(p.qs):
        x[..., j, :] = words(*lead, p.n, lo=0, hi=q)
    return x


def call(case):
    c = CASES[case]
    if case in ("lwe", "dp4a"):
        D1, D0, B = c
        db, q = words(D1 * D0, lo=-128, hi=128, dtype=torch.int8), words(B * D0)
        out = torch.empty(B * D1, dtype=torch.int32, device="cuda")
        path = g.PIR_LWE_TENSOR if case == "lwe" else g.PIR_LWE_SIMT
        return lambda: g.pir_lwe_answer(db, D1, D0, q, B, out, path=path)
    if case.startswith("ntt"):
        n, L, count = c
        p = g.pir_make_params(n, 16, 1, 1, L)
        x = residues(p, count)
        return lambda: g.ntt_inv(p, g.ntt_fwd(p, x))
    if case == "expand":
        n, L, levels, ell, B = c
        p = g.pir_make_params(n, 16, 1 << levels, 4, L)
        ex = g.pir_expander_create(p, levels, ell, residues(p, levels, ell, 2))
        q, out = residues(p, B, 2), torch.empty(B, 1 << levels, 2, L, n, dtype=torch.int32, device="cuda")
        return lambda: g.pir_expand(ex, q, B, 1 << levels, out)
    layout, n, log2p, D1, D2, B, tile = c
    p = g.pir_make_params(n, log2p, D1, D2, 2)
    layouts = {"plain": g.PIR_LAYOUT_PLAIN, "limb": g.PIR_LAYOUT_LIMB, "tensor": g.PIR_LAYOUT_TENSOR}
    db = g.pir_setup_db(p, words(D1 * D2 * n * log2p // 8, lo=0, hi=256, dtype=torch.uint8), layouts[layout])
    q, out = residues(p, B, D1, 2), torch.empty(B, D2, 2, 2, n, dtype=torch.int32, device="cuda")
    return lambda: g.pir_answer_ex(db, q, B, out, tile=tile)


if __name__ == "__main__":
    run = call(sys.argv[1])
    for _ in range(3):
        run()
    torch.cuda.synchronize()
    g.pir_check_device()
    print("ok")
