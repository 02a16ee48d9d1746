"""The staged scan in the shapes that it is chosen for, and its stall test on one that it is not."""
import pytest

pytest.importorskip("torch")

import paper_2606_11536_gb300 as g
from test_gpu_scan import answers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D1,D2,B", [
    (64, 256, 1), (86, 192, 1), (200, 212, 1),     # one quad of columns a lane
    (72, 456, 1), (64, 512, 1), (301, 500, 1),     # two
    (128, 256, 2), (171, 192, 2), (500, 244, 2),   # two queries
])
def test_staged_shapes_equal_gemv(D1, D2, B):
    if B == 1:
        assert g.pir_gemm_choice(g.PIR_LAYOUT_PLAIN, D1, D2, B) == 7
    scan, want = answers(2048, 2, D1, D2, B, (7, B))
    assert scan.equal(want)
    scan, want = answers(2048, 1, D1, D2, B, (7, B), k_chunk=D1 - 1)
    assert scan.equal(want)


def test_stall_on_a_shape_of_the_direct_scan():
    import torch

    p = g.pir_make_params(2048, 8, 20, 300, 1)
    db = g.pir_setup_db(p, torch.zeros(20 * 300 * 2048, dtype=torch.uint8, device="cuda"))
    try:
        q = torch.zeros(4, 20, 2, 1, 2048, dtype=torch.int32, device="cuda")
        r = torch.empty(4, 300, 2, 1, 2048, dtype=torch.int32, device="cuda")
        g.pir_answer_ex(db, q, 4, r, tile=7, flags=g.PIR_ANSWER_TEST_STALL)
        with pytest.raises(g.PirError) as ei:
            g.pir_check_device()
        assert ei.value.status == 5
        g.pir_answer_ex(db, q, 4, r, tile=7)
        assert int(r.abs().sum()) == 0
        g.pir_check_device()
    finally:
        g.pir_free_db(db)
