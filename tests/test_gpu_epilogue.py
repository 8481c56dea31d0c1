"""Leaf output chunks (32 x 32, staged by rows) at their edges: ragged rows and
columns, C on and off the 16-byte grid, alpha and beta, nothing written around C."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 1), (31, 33), (33, 31), (128, 32), (129, 257), (160, 290), (300, 64), (257, 515)])
@pytest.mark.parametrize("off,pad", [(0, 0), (0, 4), (1, 3), (4, 5)])
@pytest.mark.parametrize("tile,d", [(128, 0), (256, 0), (512, 0), (512, 2)])
def test_output_chunks_exact(m, n, off, pad, tile, d):
    import torch
    from paper_1205_2927_gb300 import fmm as F
    g = torch.Generator(device="cuda").manual_seed(m * 1000 + n)
    k = 72
    ints = lambda r, c, lim: torch.randint(-lim, lim + 1, (r, c), generator=g, device="cuda").float()
    A, B = ints(m, k, 3), ints(k, n, 3)
    ldc = n + pad
    buf = torch.full((m * ldc + off + 64,), float("nan"), device="cuda")
    C = torch.as_strided(buf, (m, n), (ldc, 1), off)
    for beta in (0.0, -2.0):
        C0 = ints(m, n, 5)
        C.copy_(C0)
        p = F.Plan(m, n, k, ldc=ldc, depth=d, leaf_tile=tile, fuse_last=1)
        p(A, B, C, alpha=0.5, beta=beta)
        torch.cuda.synchronize()
        assert p.device_status() == 0
        assert torch.equal(C.double(), 0.5 * (A.double() @ B.double()) + beta * C0.double())
        p.close()
    C.fill_(float("nan"))
    assert bool(torch.isnan(buf).all())   # nothing outside the view was written
