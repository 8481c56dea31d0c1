"""Each order of a host-resident root's products, where the sizes of A, B and C and beta
decide it: exact on small integers, and C leaves early where C is what moves."""
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# the first order: C no larger than the inputs, or with beta, or by SM copies; the second:
# C the largest (1.2 times the inputs at k = 580 of 1500 x 1300)
@pytest.mark.parametrize("k,beta,how", [(1500, 0.0, "engine"), (590, 0.0, "engine"), (570, 0.0, "engine"),
                                        (72, 0.0, "engine"), (72, -0.5, "engine"), (72, 0.0, "sm")])
def test_orders_exact(k, beta, how):
    import torch
    from paper_1205_2927_gb300 import fmm
    m, n = 1500, 1300
    A, B, C0 = I.small_int((m, k), 91, r=2), I.small_int((k, n), 92, r=2), I.small_int((m, n), 93, r=4)
    hA, hB, hC = (torch.from_numpy(x).pin_memory() for x in (A, B, C0))
    p = fmm.Plan(m, n, k, depth=1, host_operands=1, host_copy=how)
    for _ in range(2):
        hC.copy_(torch.from_numpy(C0))
        p(hA, hB, hC, alpha=2.0, beta=beta)
        torch.cuda.synchronize()
        assert p.device_status() == 0
    p.close()
    ref = 2.0 * (torch.from_numpy(A).cuda().double() @ torch.from_numpy(B).cuda().double())
    ref += beta * torch.from_numpy(C0).cuda().double()
    assert torch.equal(hC.cuda(), ref.float())


def test_large_c_leaves_early():
    # 0.94 ms; 1.07 with the first quadrant of C behind six of the eight input quadrants.
    # The link alone takes 0.13 ms in before that and 0.75 out.
    import torch
    from paper_1205_2927_gb300 import fmm
    m = n = 6000
    k = 750
    A, B, C = (torch.zeros(s).pin_memory() for s in ((m, k), (k, n), (m, n)))
    p = fmm.Plan(m, n, k, depth=1, host_operands=1, host_copy="engine")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ms = []
    for _ in range(8):
        e[0].record()
        for _ in range(5):
            p(A, B, C)
        e[1].record()
        torch.cuda.synchronize()
        ms.append(e[0].elapsed_time(e[1]) / 5)
    p.close()
    # against C's way out alone, by the same engines
    D, out = torch.zeros(m, n, device="cuda"), []
    for _ in range(6):
        e[0].record()
        for _ in range(5):
            C.copy_(D, non_blocking=True)
        e[1].record()
        torch.cuda.synchronize()
        out.append(e[0].elapsed_time(e[1]) / 5)
    assert min(ms[1:]) <= 1.38 * min(out), (ms, out)
