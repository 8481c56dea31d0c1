"""Host-resident plans at depth 0: panels of the larger operand and of C, each
multiplied while the next arrives, give the device-resident plan's result."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1205_2927_gb300 import fmm
    return fmm


# rows split / columns split; panels of whole tiles and a remainder of one row or
# column; the fewest and the most panels; rows that no 16-byte load may touch
@pytest.mark.parametrize("m,n,k,prec,how", [(1536, 1024, 300, "fp32", "engine"), (1537, 1030, 333, "fp32", "sm"),
                                            (1100, 2049, 515, "fp32", "sm"), (1029, 4100, 260, "bf16x3", "engine"),
                                            (4357, 4099, 65, "tf32", "sm"), (1300, 1290, 200, "fp16x3", "engine"),
                                            (6145, 6143, 32, "fp32", "engine")])
@pytest.mark.parametrize("beta", [0.0, -0.5])
def test_panels_equal_device_plan(F, m, n, k, prec, how, beta):
    import torch
    A, B = I.uniform((m, k), 61 + m), I.uniform((k, n), 62 + n)
    C0 = I.uniform((m, n), 63)
    hA, hB, hC = (torch.from_numpy(x).pin_memory() for x in (A, B, C0))
    p = F.Plan(m, n, k, depth=0, precision=prec, leaf_tile=512, host_operands=1, host_copy=how)
    for _ in range(2):   # the second call meets the first one's buffers
        hC.copy_(torch.from_numpy(C0))
        p(hA, hB, hC, alpha=0.75, beta=beta)
        torch.cuda.synchronize()
        assert p.device_status() == 0
    p.close()
    # the host plan's own buffers have rows of whole float4s (which decides how A's
    # high part is rounded): the device plan gets the same layout
    up = lambda x: (x + 3) // 4 * 4

    def padded(X):
        t = torch.zeros(X.shape[0], up(X.shape[1]), device="cuda")
        t[:, :X.shape[1]] = torch.from_numpy(X)
        return t
    d = F.Plan(m, n, k, lda=up(k), ldb=up(n), ldc=up(n), depth=0, precision=prec, leaf_tile=512)
    dA, dB, dC = padded(A), padded(B), padded(C0)
    F.fmm_gemm(d.handle, 0.75, dA.data_ptr(), dB.data_ptr(), beta, dC.data_ptr())
    torch.cuda.synchronize()
    assert d.device_status() == 0
    d.close()
    assert np.array_equal(hC.numpy(), dC[:, :n].cpu().numpy())


@pytest.mark.parametrize("m,n", [(1500, 1300), (14200, 14100)])   # each order of the root's products
@pytest.mark.parametrize("beta", [0.0, -0.5])
def test_root_orders_exact(F, m, n, beta):
    import torch
    k = 72
    A, B, C0 = I.small_int((m, k), 91, r=2), I.small_int((k, n), 92, r=2), I.small_int((m, n), 93, r=4)
    hA, hB, hC = (torch.from_numpy(x).pin_memory() for x in (A, B, C0))
    p = F.Plan(m, n, k, depth=1, host_operands=1, host_copy="engine")
    p(hA, hB, hC, alpha=2.0, beta=beta)
    torch.cuda.synchronize()
    assert p.device_status() == 0
    p.close()
    ref = 2.0 * (torch.from_numpy(A).cuda().double() @ torch.from_numpy(B).cuda().double())
    ref += beta * torch.from_numpy(C0).cuda().double()
    assert torch.equal(hC.cuda(), ref.float())
