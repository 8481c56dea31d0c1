"""Depth-0 pair launches whose last tiles go out in column parts: every element is the
one that the same product gives as part of a wider one whose plan names its tile."""
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# tiles on 76 pairs: 16 (quarters), 20 and 36 (halves), 76 + 4 and 76 + 20, 2 * 76 + 17,
# 3 * 76 + 12; M, N and K off every boundary, the last tile column 1, 29, 65 or 130 wide
# (parts with no columns of their own)
@pytest.mark.parametrize("m,n,k", [(1024, 1024, 64), (1280, 1024, 333), (1283, 1536 - 126, 200),
                                   (2048, 10 * 256 - 255, 33), (2045, 12 * 256 - 227, 1000),
                                   (13 * 256, 13 * 256 - 191, 161), (16 * 256, 15 * 256 - 126, 96)])
@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16x3", "fp16x3"])
def test_tail_parts_equal_whole_tiles(m, n, k, prec):
    import torch
    from paper_1205_2927_gb300 import fmm
    wide = n + 256   # named tiles: whole ones
    A = torch.from_numpy(I.uniform((m, k), 81 + m)).cuda()
    B = torch.zeros((k, wide), device="cuda")
    B[:, :n] = torch.from_numpy(I.uniform((k, n), 82 + n)).cuda()
    C0 = torch.from_numpy(I.uniform((m, n), 83)).cuda()

    def run(cols, beta, tile):
        C = torch.zeros((m, cols), device="cuda")
        C[:, :n] = C0
        p = fmm.Plan(m, cols, k, depth=0, precision=prec, leaf_tile=tile)
        p(A, B[:, :cols].contiguous(), C, alpha=0.5, beta=beta)
        torch.cuda.synchronize()
        assert p.device_status() == 0
        p.close()
        return C[:, :n]
    assert torch.equal(run(n, -2.0, 0), run(wide, -2.0, 512))
