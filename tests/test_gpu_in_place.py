"""C in the memory of an operand (small products, which one launch computes from the
caller's A and B; depth-0 plans; host-resident panels) gives the bits that a C of its
own gives, and column blocks of one buffer, which share nothing, keep their route."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1205_2927_gb300 import fmm
    return fmm


def _views(m, n, k, over, shift, host=False):
    """A, B and a C that starts `shift` floats into A (over = "A") or B, in one buffer each;
    and the values of A, B and C before the call."""
    import torch
    new = (lambda c: torch.empty(c).pin_memory()) if host else (lambda c: torch.empty(c, device="cuda"))
    bufs = {"A": new(m * k + m * n + shift), "B": new(k * n + m * n + shift)}
    A, B = bufs["A"][: m * k].view(m, k), bufs["B"][: k * n].view(k, n)
    C = bufs[over][shift: shift + m * n].view(m, n)
    C.copy_(torch.from_numpy(I.uniform((m, n), 3)))
    A.copy_(torch.from_numpy(I.uniform((m, k), 1)))
    B.copy_(torch.from_numpy(I.uniform((k, n), 2)))
    return A, B, C, A.clone(), B.clone(), C.clone()


CASES = [(256, 256, 256, 0), (300, 300, 300, 0), (1000, 1000, 1000, 0), (300, 516, 300, 4), (516, 300, 516, 1024)]


@pytest.mark.parametrize("m,n,k,shift", CASES)
@pytest.mark.parametrize("over", ["A", "B"])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_static(F, m, n, k, shift, over, beta):
    import torch
    A, B, C, A0, B0, C0 = _views(m, n, k, over, shift)
    F.fmm_gemm_static(A0, B0, C0, alpha=0.75, beta=beta)
    F.fmm_gemm_static(A, B, C, alpha=0.75, beta=beta)
    assert F.fmm_gemm_static_status() == 0
    assert torch.equal(C, C0)


@pytest.mark.parametrize("m,n,k,shift", CASES + [(1536, 1100, 260, 0)])
@pytest.mark.parametrize("over", ["A", "B"])
@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16x3", "fp16x3"])
def test_plans(F, m, n, k, shift, over, prec):
    import torch
    A, B, C, _, _, _ = _views(m, n, k, over, shift)
    ints = lambda t, seed: t.copy_(torch.from_numpy(I.small_int(tuple(t.shape), seed, r=3)))
    ints(C, 6), ints(A, 4), ints(B, 5)      # exact by every route
    A0, B0, C0 = A.double(), B.double(), C.double()
    p = F.Plan(m, n, k, depth=0, precision=prec)
    p(A, B, C, alpha=1.0, beta=-2.0)
    torch.cuda.synchronize()
    assert p.device_status() == 0
    p.close()
    assert torch.equal(C.double(), A0 @ B0 - 2.0 * C0)


# rows and columns split; C's rows longer than A's, so that it runs ahead of the panels
@pytest.mark.parametrize("m,n,k,shift", [(1600, 1100, 300, 0), (1100, 1600, 300, 0), (1300, 1290, 1300, 7)])
@pytest.mark.parametrize("over", ["A", "B"])
def test_host_panels(F, m, n, k, shift, over):
    import torch
    A, B, C, A0, B0, C0 = _views(m, n, k, over, shift, host=True)
    own = [t.pin_memory() for t in (A0, B0, C0)]
    p = F.Plan(m, n, k, depth=0, leaf_tile=512, host_operands=1, host_copy="engine")
    for operands in (own, (A, B, C)):
        p(*operands, alpha=0.75, beta=0.5)
        torch.cuda.synchronize()
        assert p.device_status() == 0
    p.close()
    assert np.array_equal(C.numpy(), own[2].numpy())


def test_column_blocks_of_one_buffer_keep_the_one_launch(F):
    import torch
    m = n = k = 256
    W = torch.zeros(m, 3 * n + 9, device="cuda")
    A, B, C = W[:, :k], W[:, k: k + n], W[:, k + n + 9:]
    A.copy_(torch.from_numpy(I.small_int((m, k), 1))), B.copy_(torch.from_numpy(I.small_int((k, n), 2)))
    p = F.Plan(m, n, k, W.stride(0), W.stride(0), W.stride(0))
    p.profile(True)
    p(A, B, C)
    torch.cuda.synchronize()
    assert p.profile_read()["launches"] == 1
    p.close()
    assert torch.equal(C.double(), A.double() @ B.double())
