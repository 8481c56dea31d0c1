"""The cost model's training step at the edges of its tiles and block counts:
gradient, moments, loss and update against the float64 oracle."""
import numpy as np
import pytest

import oracle.fmm_oracle as O

pytestmark = pytest.mark.gpu


# 1..33: one block (the workspace of 33 samples holds one row of sums); 73: two
# blocks; 14593: 457 tiles, two per block, the last block with one sample
@pytest.mark.parametrize("n", [1, 18, 32, 33, 73, 14593])
def test_train_step_matches_oracle(n):
    import torch
    from paper_1205_2927_gb300 import fmm as F
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 6)).astype(np.float32)
    t = (0.5 * X[:, 0] - X[:, 3] * X[:, 1] + 0.2).astype(np.float32)
    theta = (rng.standard_normal(O.MLP_NPARAM) * 0.3).astype(np.float32)
    m0 = (rng.standard_normal(O.MLP_NPARAM) * 1e-2).astype(np.float32)
    v0 = (rng.random(O.MLP_NPARAM) * 1e-2 + 1e-3).astype(np.float32)
    p, m, v = (torch.from_numpy(a.copy()).cuda() for a in (theta, m0, v0))
    g, loss = torch.empty_like(p), torch.zeros(1, device="cuda")
    ws = torch.empty(F.mlp_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    F.fmm_mlp_train_step(p, m, v, 7, 1e-2, torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda(), ws, grad_out=g,
                         loss_out=loss)
    lref, gref = O.mlp_grad(theta.astype(np.float64), X.astype(np.float64), t.astype(np.float64))
    pref, mref, vref = O.adam_step(theta.astype(np.float64), m0.astype(np.float64), v0.astype(np.float64), gref, 7, 1e-2)
    # fp32 sums of at most 32 samples in series, then of at most 30 rows: well under
    # 1e-5 of the largest entry
    assert np.max(np.abs(g.cpu().numpy() - gref)) <= 1e-5 * np.abs(gref).max()
    assert float(loss.item()) == pytest.approx(lref, rel=1e-5)
    assert np.allclose(m.cpu().numpy(), mref, rtol=1e-5, atol=1e-6 * np.abs(gref).max())
    assert np.allclose(v.cpu().numpy(), vref, rtol=1e-4, atol=1e-7 * np.abs(gref).max() ** 2)
    assert np.allclose(p.cpu().numpy(), pref, rtol=1e-5, atol=1e-6)
