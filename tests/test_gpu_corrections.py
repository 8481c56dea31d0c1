"""FP32 leaves on CTA pairs: one TF32 product plus bf16 correction products.

Exactness where every product is exact (one side's lo parts against a sparse
small side), at row lengths around the 32-column lines of the correction plane
and in every pass that writes it; and no more error against float64 than the
three TF32 products (single-CTA tiles) at the limits of the rule that picks it.
"""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmm():
    from paper_1205_2927_gb300 import fmm as F
    return F


def _lo_operand(shape, seed):
    """Integers a * 4096 + b, |a| <= 2, b in {-1, 0, 1}: exact as a TF32 hi of one
    or two bits and a one-bit lo, and so are sums of a few of them."""
    g = np.random.default_rng(seed)
    return (g.integers(-2, 3, shape) * 4096 + g.integers(-1, 2, shape)).astype(np.float32)


def _sparse(k, n, seed):
    """Two +-1 per column, one of them in the last rows."""
    g = np.random.default_rng(seed)
    B = np.zeros((k, n), np.float32)
    for j in range(n):
        B[g.integers(0, k), j] = g.choice([-1, 1])
        B[k - 1 - j % min(k, 40), j] = g.choice([-1, 1])
    return B


# depth 0 (k around multiples of 32 and 4), depth 1, depth 2 fused and not
@pytest.mark.parametrize("m,k,n,d", [(256, 192, 256, 0), (300, 193, 260, 0), (260, 223, 300, 0), (513, 1001, 257, 0),
                                     (256, 6144, 256, 0), (600, 1030, 520, 1), (512, 2047, 512, 1),
                                     (1024, 4100, 1024, 2), (1100, 4096, 900, 2)])
@pytest.mark.parametrize("side", ["A", "B"])
def test_corrections_exact(fmm, m, k, n, d, side):
    import torch
    if side == "A":
        A, B = _lo_operand((m, k), m + k), _sparse(k, n, n + k)
    else:
        A, B = _sparse(k, m, m + k).T.copy(), _lo_operand((k, n), n + k)
    ref = torch.from_numpy(A).cuda().double() @ torch.from_numpy(B).cuda().double()
    for off in (0, 1):   # off 1: A off the 16-byte grid, both of its planes written
        dA = torch.empty(m * k + off, device="cuda")[off:].view(m, k)
        dA.copy_(torch.from_numpy(A))
        C0 = torch.full((m, n), 3.0, device="cuda")
        p = fmm.Plan(m, n, k, depth=d, leaf_tile=512)
        p(dA, torch.from_numpy(B).cuda(), C0, alpha=1.0, beta=-1.0)
        torch.cuda.synchronize()
        assert p.device_status() == 0
        assert torch.equal(C0.double(), ref - 3.0)
        p.close()


def test_corrections_batched_exact(fmm):
    # one launch over problems of both FP32 plane forms, at depths 0 to 2
    import torch
    shapes = [(256, 40, 300), (130, 191, 70), (300, 192, 260), (64, 777, 513), (257, 1100, 255), (1024, 4096, 1028)]
    As = [torch.from_numpy(_lo_operand((m, k), i)).cuda() for i, (m, k, n) in enumerate(shapes)]
    Bs = [torch.from_numpy(_sparse(k, n, 50 + i)).cuda() for i, (m, k, n) in enumerate(shapes)]
    for cutoff in (2048, 256):
        Cs = [torch.empty((m, n), device="cuda") for m, k, n in shapes]
        p = fmm.BatchedPlan(As, Bs, Cs, cutoff=cutoff)
        p.run()
        torch.cuda.synchronize()
        assert max(p.info()["depths"]) == (0 if cutoff == 2048 else 2)
        for A, B, C in zip(As, Bs, Cs):
            assert torch.equal(C.double(), A.double() @ B.double())
        p.close()


@pytest.mark.parametrize("m,k,n,d", [(768, 192, 1024, 0), (512, 6144, 512, 0), (1024, 1024, 1024, 1),
                                     (512, 12288, 512, 1), (1024, 4096, 1024, 2), (1024, 12288, 1024, 2)])
@pytest.mark.parametrize("dist", ["uniform", "normal", "loguniform"])
def test_corrections_no_less_exact(fmm, m, k, n, d, dist):
    import torch
    A, B = (torch.from_numpy(x).cuda() for x in I.operands(m, k, n, 900 + k + d, dist))
    ref = A.double() @ B.double()
    err = {}
    for tile in (512, 256):
        p = fmm.Plan(m, n, k, depth=d, leaf_tile=tile)
        err[tile] = float((p(A, B).double() - ref).norm() / ref.norm())
        p.close()
    assert err[512] <= err[256], err
