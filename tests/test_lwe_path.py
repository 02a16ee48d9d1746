"""The scalar-HE product's choice of path (host arithmetic, no GPU): tensor-map coordinates are
signed 32-bit, so databases whose rows reach 2^31 are answered on the CUDA cores."""
import pytest

import paper_2606_11536_gb300 as g

LIMIT = 1 << 31


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2606_11536_gb300 import build
    build.build()


@pytest.mark.parametrize("path", [g.PIR_LWE_TENSOR, g.PIR_LWE_AUTO])
@pytest.mark.parametrize("B", [1, 8, 33])
def test_rows_the_tensor_maps_reach(path, B):
    for D1 in (LIMIT - 256, LIMIT - 255, LIMIT - 1, LIMIT):
        assert g.pir_lwe_path(D1, 16, B, path) == g.PIR_LWE_TENSOR, D1
    for D1 in (LIMIT + 1, LIMIT + 256, (1 << 32) - 256, (1 << 32) - 1):
        assert g.pir_lwe_path(D1, 16, B, path) == g.PIR_LWE_SIMT, D1


def test_the_cuda_core_path_stays_itself():
    for D1 in (1, 4096, LIMIT, LIMIT + 1):
        assert g.pir_lwe_path(D1, 1024, 32, g.PIR_LWE_SIMT) == g.PIR_LWE_SIMT


def test_arguments():
    for bad in ((0, 16, 1, 0), (1, 0, 1, 0), (1, 16, 0, 0), (1, 16, 1, 3)):
        with pytest.raises(g.PirError) as ei:
            g.pir_lwe_path(*bad)
        assert ei.value.status == 1


@pytest.mark.gpu
def test_rows_past_2_31():
    """Rows on both sides of 2^31 (34 GiB of records, one query) against the definition."""
    import numpy as np
    import torch

    D1, D0 = LIMIT + 515, 16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    db = torch.empty(D1 * D0, dtype=torch.int8, device="cuda")
    step = 1 << 32
    for i in range(0, D1 * D0, step):
        part = db[i:i + step]
        part.copy_(torch.randint(-128, 128, (part.numel(),), generator=gen, dtype=torch.int8, device="cuda"))
    q = torch.randint(-2**31, 2**31 - 1, (D0,), generator=gen, dtype=torch.int32, device="cuda")
    out = torch.zeros(D1, dtype=torch.int32, device="cuda")
    g.pir_lwe_answer(db, D1, D0, q, 1, out)
    rows = np.r_[0:256, LIMIT - 256:LIMIT + 515, np.random.default_rng(1).integers(0, D1, 4096)]
    idx = torch.from_numpy(rows).cuda()
    A = db.view(D1, D0)[idx].cpu().numpy().astype(np.int64)
    want = (A @ q.cpu().numpy().astype(np.int64)) & 0xFFFFFFFF  # |sum| < 2^42
    got = out[idx].cpu().numpy().view(np.uint32).astype(np.int64)
    g.pir_check_device()
    del db, out
    torch.cuda.empty_cache()
    assert np.array_equal(got, want)
