"""Leaf launches over a few waves of tiles, with a grid that fills every wave:
integer operands, exact results."""
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# one tile over a wave; two waves and a remainder; four waves; five (the full grid)
@pytest.mark.parametrize("m,n", [(256 * 7, 256 * 11), (2305, 4097), (4096, 4864), (4096, 5120)])
@pytest.mark.parametrize("prec,tile", [("fp32", 512), ("fp32", 256), ("tf32", 512), ("tf32", 256), ("bf16x3", 512)])
def test_wave_grid_exact(m, n, prec, tile):
    import torch
    from paper_1205_2927_gb300 import fmm
    k = 1024
    A, B = I.small_int((m, k), 7000 + m, r=2), I.small_int((k, n), 7100 + n, r=2)
    C = torch.full((m, n), float("nan"), device="cuda")
    p = fmm.Plan(m, n, k, depth=0, precision=prec, leaf_tile=tile)
    p(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C)
    torch.cuda.synchronize()
    assert p.device_status() == 0
    p.close()
    ref = (torch.from_numpy(A).cuda().double() @ torch.from_numpy(B).cuda().double()).float()
    assert torch.equal(C, ref)
