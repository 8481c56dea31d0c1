"""The exhaustive planner on small products: it times depth 0 as the plan runs it, so
where one launch takes half of any level's time, that launch is what the plan is."""
import pytest

pytestmark = pytest.mark.gpu


# one launch and the fastest level, measured (us): 11 and 22, 12.5 and 27, 14 and 24, 9 and 17,
# 9.9 and 19
@pytest.mark.parametrize("prec,m,n,k", [("fp32", 768, 768, 768), ("fp32", 1024, 512, 1024), ("fp32", 700, 515, 901),
                                        ("tf32", 768, 768, 768), ("tf32", 1024, 512, 1024)])
def test_picks_the_one_launch(prec, m, n, k):
    import torch
    from paper_1205_2927_gb300 import fmm
    A, B = torch.rand(m, k, device="cuda") - 0.5, torch.rand(k, n, device="cuda") - 0.5
    p = fmm.Plan(m, n, k, precision=prec, planner="exhaustive")
    p.profile(True)
    C = p(A, B)
    torch.cuda.synchronize()
    assert p.device_status() == 0
    assert p.info["depth"] == 0 and p.profile_read()["launches"] == 1
    p.close()
    ref = A.double() @ B.double()
    assert float((C.double() - ref).norm() / ref.norm()) < (2e-3 if prec == "tf32" else 2e-5)
