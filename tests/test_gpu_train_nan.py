"""A target that is NaN shows in every entry of the last layer's gradient, also of
units that its sample leaves at zero (0 x NaN)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [20, 100])   # one block, and several
def test_nan_target_reaches_every_output_weight(n):
    import torch
    from paper_1205_2927_gb300 import fmm as F
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 6)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    t[n // 3] = np.nan
    p = torch.from_numpy((rng.standard_normal(F.NPARAM) * 0.3).astype(np.float32)).cuda()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    g, loss = torch.empty_like(p), torch.zeros(1, device="cuda")
    ws = torch.empty(F.mlp_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    F.fmm_mlp_train_step(p, m, v, 1, 0.0, torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda(), ws, grad_out=g,
                         loss_out=loss)
    w3, b3 = g[4608:4672], g[4672]
    assert bool(torch.isnan(w3).all()) and bool(torch.isnan(b3)) and bool(torch.isnan(loss).all())
    assert not bool(torch.isnan(g[:4608]).all())   # hidden units that are off stay out of it
