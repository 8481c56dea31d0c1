"""FP32 products whose corrections run in bf16 (CTA-pair leaves of a range of
lengths): infinities, and the same bits at any alignment of the operands."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

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


def _placed(X, off, pad):
    """X at an offset of `off` floats, rows `pad` floats longer."""
    import torch
    m, k = X.shape
    t = torch.zeros(off + m * (k + pad), device="cuda")[off:].view(m, k + pad)
    t[:, :k] = torch.from_numpy(X)
    return t[:, :k]


# lengths around the 32-column lines; depth 0 with bf16 corrections (k from 192 on) and
# without, and a level of each
@pytest.mark.parametrize("m,k,n,d", [(300, 160, 260, 0), (300, 192, 260, 0), (258, 516, 300, 0), (513, 1004, 257, 0),
                                     (600, 1032, 520, 1), (1024, 4100, 1028, 2)])
def test_same_bits_at_any_alignment(fmm, m, k, n, d):
    A, B = I.normal((m, k), m + k), I.normal((k, n), k + n)
    got = []
    for off, pad in ((0, 0), (1, 0), (0, 3)):   # on the 16-byte grid; off it by its start; by its rows
        dA, dB = _placed(A, off, pad), _placed(B, off, pad)
        p = fmm.Plan(m, n, k, k + pad, n + pad, n, depth=d, leaf_tile=512)
        got.append(p(dA, dB).clone())
        assert p.device_status() == 0
        p.close()
    assert all((g == got[0]).all() for g in got[1:])


def test_batched_same_bits_at_any_alignment(fmm):
    import torch
    shapes = [(256, 160, 300), (130, 192, 72), (300, 516, 260), (257, 1004, 256)]
    got = []
    for off, pad in ((0, 0), (1, 0), (0, 3)):
        As = [_placed(I.normal((m, k), i), off, pad) for i, (m, k, n) in enumerate(shapes)]
        Bs = [_placed(I.normal((k, n), 9 + i), off, pad) for i, (m, k, n) in enumerate(shapes)]
        Cs = [torch.empty((m, n), device="cuda") for m, k, n in shapes]
        p = fmm.BatchedPlan(As, Bs, Cs)
        p.run()
        torch.cuda.synchronize()
        p.close()
        got.append(Cs)
    for other in got[1:]:
        assert all(torch.equal(x, y) for x, y in zip(got[0], other))


def test_host_resident_equals_device_resident_off_the_grid(fmm):
    import torch
    m, n, k = 1537, 1030, 333
    A, B = I.normal((m, k), 71), I.normal((k, n), 72)
    hA, hB, hC = (torch.from_numpy(x).pin_memory() for x in (A, B, np.zeros((m, n), np.float32)))
    p = fmm.Plan(m, n, k, depth=0, leaf_tile=512, host_operands=1)
    p(hA, hB, hC)
    torch.cuda.synchronize()
    p.close()
    dC = fmm.Plan(m, n, k, depth=0, leaf_tile=512)(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda())
    assert torch.equal(hC.cuda(), dC)
