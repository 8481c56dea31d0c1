"""Overlapping a pass with the end of the one before it must not cost more than it
hides: calls in a row take no longer than the phases of a call take one by one (events
between the phases keep their launches apart)."""
import pytest

pytestmark = pytest.mark.gpu


# depth 3 on ragged sizes: a leaf launch of short tiles, post-additions of 35 and of 3565
# blocks, pre-additions by levels (TF32) and at once
@pytest.mark.parametrize("m,n,k,prec,tile", [(269, 277, 3195, "fp32", 128), (5700, 4441, 312, "tf32", 512)])
def test_calls_in_a_row_take_no_longer_than_their_phases(m, n, k, prec, tile):
    import torch
    from paper_1205_2927_gb300 import fmm
    A, B = torch.rand(m, k, device="cuda") - 0.5, torch.rand(k, n, device="cuda") - 0.5
    C = torch.empty(m, n, device="cuda")
    p = fmm.Plan(m, n, k, depth=3, precision=prec, leaf_tile=tile)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    row, apart = [], []
    for _ in range(6):
        e[0].record()
        for _ in range(30):
            p(A, B, C)
        e[1].record()
        torch.cuda.synchronize()
        row.append(e[0].elapsed_time(e[1]) / 30)
        p.profile(True)
        for _ in range(30):
            p(A, B, C)
        torch.cuda.synchronize()
        q = p.profile_read()
        p.profile(False)
        apart.append((q["pre_ms"] + q["leaf_ms"] + q["post_ms"]) / 30)
    p.close()
    assert min(row[1:]) <= 1.04 * min(apart[1:]), (row, apart)
