"""Operand maxima of FP16x3 calls: one element decides the scale, wherever it lies."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# the largest element at the first and last position, across 32 x 128 blocks and
# ragged edges, on rows with and without 16-byte loads; plan and batch.  Its value
# 3e4 times the rest's integers overflows fp16 unless the scale saw it
@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (33, 129, 131), (64, 256, 128), (500, 1001, 130)])
@pytest.mark.parametrize("side", ["A", "B"])
@pytest.mark.parametrize("where", [0, -1])
def test_scale_sees_the_largest_element(m, k, n, side, where):
    import torch
    from paper_1205_2927_gb300 import fmm
    A, B = I.small_int((m, k), 500 + m, r=2), I.small_int((k, n), 600 + n, r=2)
    (A if side == "A" else B).flat[where] = 2.0 ** 20
    ref = (A.astype(np.float64) @ B.astype(np.float64)).astype(np.float32)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    p = fmm.Plan(m, n, k, depth=0, precision="fp16x3", leaf_tile=256)
    C = torch.full((m, n), float("nan"), device="cuda")
    p(dA, dB, C)
    other = torch.from_numpy(I.small_int((200, 300), 7, r=2)).cuda()
    Cs = [torch.full((200, 200), float("nan"), device="cuda"), torch.full((m, n), float("nan"), device="cuda"),
          torch.full((200, 200), float("nan"), device="cuda")]
    bp = fmm.BatchedPlan([other, dA, other], [other.T.contiguous(), dB, other.T.contiguous()], Cs, precision="fp16x3")
    bp.run()
    torch.cuda.synchronize()
    p.close()
    o = other.double()
    assert np.array_equal(C.cpu().numpy(), ref)
    assert np.array_equal(Cs[1].cpu().numpy(), ref)
    assert torch.equal(Cs[0], (o @ o.T).float()) and torch.equal(Cs[2], (o @ o.T).float())
