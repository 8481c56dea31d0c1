"""fp64 residual: row counts around the rows a block takes, 16-byte rows and
others, and values that the integer widening leaves to the conversion."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1215, 260), (1216, 260), (1219, 1028), (2431, 259), (2432, 259), (2439, 1027),
                                       (1, 3), (5, 1024)])
def test_row_and_column_edges_exact(rows, cols):
    import torch
    from paper_1205_2927_gb300 import fmm as F
    A, B = I.small_int((rows, cols), rows, r=3), I.small_int((cols, cols), cols, r=3)
    C, x = I.small_int((rows, cols), rows + 1, r=3), I.small_int((cols,), 9, r=5)
    r = F.fmm_residual(*(torch.from_numpy(t).cuda() for t in (A, B, C, x)), fp64=True)
    want = C.astype(np.float64) @ x - A.astype(np.float64) @ (B.astype(np.float64) @ x)
    assert np.array_equal(r.cpu().numpy(), want)


@pytest.mark.parametrize("cols", [64, 61])
def test_special_values(cols):
    # one value per row of C beside zeros, A = 0: r is that value times x, exactly
    import torch
    from paper_1205_2927_gb300 import fmm as F
    vals = np.array([0.0, -0.0, 1e-45, -3e-40, 1.1754944e-38, 1.1754942e-38, 3.4028235e38, -3.4028235e38, np.inf,
                     -np.inf, np.nan, 1.0, -1.5, 6.1e-5, 65504.0], np.float32)
    rows = 2448
    C = np.zeros((rows, cols), np.float32)
    C[np.arange(rows), np.arange(rows) % cols] = vals[np.arange(rows) % len(vals)]
    x = np.where(np.arange(cols) % 3 == 0, -1.0, 1.5).astype(np.float32)
    A, B = np.zeros((rows, 4), np.float32), np.ones((4, cols), np.float32)
    r = F.fmm_residual(*(torch.from_numpy(t).cuda() for t in (A, B, C, x)), fp64=True).cpu().numpy()
    want = vals[np.arange(rows) % len(vals)].astype(np.float64) * x[np.arange(rows) % cols].astype(np.float64)
    assert np.array_equal(r, want, equal_nan=True)
