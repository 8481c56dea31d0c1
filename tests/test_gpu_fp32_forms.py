"""FP32 products whose corrections run in bf16 (CTA-pair leaves of a range of
lengths): infinities."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmm():
    from paper_1205_2927_gb300 import fmm as F
    return F


@pytest.mark.parametrize("off", [0, 1])   # 1: A off the 16-byte grid
def test_infinities_as_ieee(fmm, off):
    import torch
    m, k, n = 300, 260, 270
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn(m * k + off, generator=g, device="cuda")[off:].view(m, k)
    B = torch.randn(k, n, generator=g, device="cuda")
    inf = float("inf")
    A[3, 5], A[140, 259], A[299, 0] = inf, -inf, inf
    B[17, 9], B[259, 269] = -inf, inf
    A[50, 17] = 0.0                      # 0 x inf
    ref = A.double() @ B.double()
    batched = torch.empty(m, n, device="cuda")
    p = fmm.BatchedPlan([A], [B], [batched])
    p.run()
    p.close()
    inf_at = torch.isinf(ref)
    assert int(inf_at.sum()) > 1000 and int(torch.isnan(ref).sum()) >= 1
    for C in (fmm.Plan(m, n, k, depth=0, leaf_tile=512)(A, B), batched):
        got = C.double()
        assert torch.equal(torch.isnan(got), torch.isnan(ref))
        assert torch.equal(torch.isinf(got), inf_at) and torch.equal(got[inf_at], ref[inf_at])
