"""That the routes which other tests compare are the ones that run: small products as
one launch in every precision, and the last wave of a depth-0 pair launch in parts."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1205_2927_gb300 import fmm
    return fmm


# launches of the one-launch route; FP16x3 finds its scales in two more
@pytest.mark.parametrize("prec,launches", [("fp32", 1), ("tf32", 1), ("bf16x3", 1), ("fp16x3", 3)])
@pytest.mark.parametrize("m,n,k", [(130, 700, 63), (700, 515, 901), (256, 1999, 257), (1100, 1030, 64)])
@pytest.mark.parametrize("pad", [0, 5])
def test_small_products_are_one_launch(F, prec, launches, m, n, k, pad):
    import torch
    A, B, C = (torch.zeros(r, c + pad, device="cuda")[:, :c] for r, c in ((m, k), (k, n), (m, n)))
    counts = {}
    for tile in (0, 256):   # left open; named, by the leaf path
        p = F.Plan(m, n, k, k + pad, n + pad, n + pad, precision=prec, leaf_tile=tile)
        p.profile(True)
        p(A, B, C)
        torch.cuda.synchronize()
        counts[tile] = p.profile_read()["launches"]
        p.close()
    assert counts[0] == launches < counts[256], counts


# 16 tiles on 76 pairs go out in 64 parts: FP32 75 us against 91, BF16x3 50 against 69
@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
def test_few_tiles_take_parts(F, prec):
    import torch
    m = n = 1024
    k = 4096
    A, B = torch.rand(m, k, device="cuda"), torch.rand(k, n, device="cuda")
    C = torch.empty(m, n, device="cuda")
    us = {}
    for tile in (0, 512):
        p = F.Plan(m, n, k, depth=0, precision=prec, leaf_tile=tile)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        runs = []
        for _ in range(6):
            e[0].record()
            for _ in range(20):
                p(A, B, C)
            e[1].record()
            torch.cuda.synchronize()
            runs.append(e[0].elapsed_time(e[1]) * 50)
        us[tile] = min(runs[1:])
        p.close()
    assert us[0] < 0.93 * us[512], us
