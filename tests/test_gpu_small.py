"""The one-launch kernel of small products: exact on small integers at the edges
of its tiles, K steps and K shares (through the entry point that always takes
it, and through plans that choose it), and no further from float64 than the leaf
path it replaces."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1205_2927_gb300 import fmm
    return fmm


def _ints(g, r, c, pad, lim=3):
    import torch
    buf = torch.full((r, c + pad), float("nan"), device="cuda")
    buf[:, :c] = torch.randint(-lim, lim + 1, (r, c), generator=g, device="cuda").float()
    return buf[:, :c]


# sizes whose choices cover tiles of 32, 64 and 128 columns and K shared by 1 to 8 CTAs
@pytest.mark.parametrize("m,n", [(1, 1), (127, 31), (128, 32), (129, 33), (300, 65), (257, 513), (1024, 1000)])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 129, 500, 1024])
@pytest.mark.parametrize("pad", [0, 3])
def test_static_exact(F, m, n, k, pad):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m * 7 + n * 3 + k)
    A, B, C = _ints(g, m, k, pad), _ints(g, k, n, pad), _ints(g, m, n, pad, 5)
    ref = 0.5 * (A.double() @ B.double()) - 2.0 * C.double()
    F.fmm_gemm_static(A, B, C, alpha=0.5, beta=-2.0)
    assert F.fmm_gemm_static_status() == 0
    assert torch.equal(C.double(), ref)
    if pad:
        assert bool(torch.isnan(C.as_strided((m, pad), (n + pad, 1), n)).all())


@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("m,n,k", [(64, 64, 5000), (130, 700, 63), (700, 515, 901), (573, 452, 2103), (256, 1999, 257),
                                   (1023, 129, 4200), (1100, 1030, 64)])
@pytest.mark.parametrize("pad", [0, 5])
def test_plans_exact_and_as_the_leaf_path(F, prec, m, n, k, pad):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A, B, C = _ints(g, m, k, pad, 2), _ints(g, k, n, pad, 2), _ints(g, m, n, pad, 5)
    ref = A.double() @ B.double() - C.double()
    p = F.Plan(m, n, k, k + pad, n + pad, n + pad, precision=prec)
    p(A, B, C, alpha=1.0, beta=-1.0)
    torch.cuda.synchronize()
    assert p.device_status() == 0 and p.info["depth"] == 0
    assert torch.equal(C.double(), ref)
    # floats: within the leaf path's own error of float64 (no longer accumulator chains)
    A.copy_(torch.rand(m, k, generator=g, device="cuda") * 2 - 1)
    B.copy_(torch.rand(k, n, generator=g, device="cuda") * 2 - 1)
    ref = A.double() @ B.double()
    err = {}
    for tile in (0, 256):
        q = F.Plan(m, n, k, k + pad, n + pad, n + pad, precision=prec, leaf_tile=tile)
        q(A, B, C)
        err[tile] = float((C.double() - ref).norm() / ref.norm())
        q.close()
    assert err[0] <= 1.001 * err[256], err   # the same products; the chains' order may differ in the last bits
    p.close()


def test_small_plan_captures_in_a_graph(F):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    A, B = _ints(g, 300, 200, 0), _ints(g, 200, 500, 0)
    C = torch.zeros(300, 500, device="cuda")
    p = F.Plan(300, 500, 200)
    p(A, B, C)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p(A, B, C)
        F.fmm_gemm_static(A, B, C, beta=1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(C.double(), 2.0 * (A.double() @ B.double()))
