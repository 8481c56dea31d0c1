"""What one term a b of an FP32 product may be off by, for operands that let it show:
a permutation, a diagonal and few non-zeros per column, where the accumulator adds
next to nothing.  In units of |a b|, from the two forms' arithmetic:

  three TF32 products (leaf tiles 128 and 256, and lengths outside the other form's):
    x = t + l with |l| < 2^-10 |x| truncated off, l to the nearest TF32 (13 bits to 11:
    2^-22), the product of both l left out (2^-20): 2^-22 for a factor that is a power
    of two, 2^-19 for any two factors
  one TF32 product with bf16 corrections (CTA-pair leaves), where l, and the value that
    meets the other side's l, are rounded to 8 bits (2^-9): 2^-19 for an element of A
    and 2^-20 for one of B (whose high part is rounded, |l| <= 2^-11) against a power of
    two; 2 (2^-19 + 2^-20) + 2^-21 < 2^-17 for any two factors

The accumulator's truncations (2^-23 of a sum, one per instruction that adds something)
come on top: with one term there are at most two additions of a low part."""
import numpy as np
import pytest

from paper_1205_2927_gb300 import inputs as I

pytestmark = pytest.mark.gpu

M, K = 520, 516
ADDS = 2 * 2.0 ** -23
# leaf tile: an element of A, of B, any two; integers below these pass unchanged (A, B)
FORMS = {512: (2.0 ** -19, 2.0 ** -20, 2.0 ** -17, 19, 20), 256: (2.0 ** -22, 2.0 ** -22, 2.0 ** -19, 22, 22)}


@pytest.fixture(scope="module")
def fmm():
    from paper_1205_2927_gb300 import fmm as F
    return F


def _product(fmm, A, B, tile, off):
    import torch
    dA = torch.empty(A.size + off, device="cuda")[off:].view(A.shape)
    dA.copy_(torch.from_numpy(A))
    p = fmm.Plan(A.shape[0], B.shape[1], A.shape[1], depth=0, leaf_tile=tile)
    got = p(dA, torch.from_numpy(B).cuda()).cpu().numpy()
    p.close()
    return got


def _selection(seed):
    g = np.random.default_rng(seed)
    P = np.zeros((K, K), np.float32)
    P[g.permutation(K), np.arange(K)] = g.choice([-1.0, 1.0, 0.5, 4.0], K)
    return P


@pytest.mark.parametrize("tile", [512, 256])
@pytest.mark.parametrize("off", [0, 1])
def test_single_terms(fmm, tile, off):
    of_a, of_b, of_ab, _, _ = FORMS[tile]
    A, P = I.normal((M, K), 5), _selection(6)
    D = np.diag(I.normal((K,), 7)).astype(np.float32)
    for X, Y, most in ((A, P, of_a), (P, A.T.copy(), of_b), (A, D, of_ab)):
        ref = X.astype(np.float64) @ Y.astype(np.float64)
        assert np.max(np.abs(_product(fmm, X, Y, tile, off) - ref) / np.abs(ref)) <= most + ADDS


@pytest.mark.parametrize("tile", [512, 256])
def test_few_terms(fmm, tile):
    # three non-zeros a column: the terms' bounds add up
    g = np.random.default_rng(8)
    A, B = I.normal((M, K), 9), np.zeros((K, M), np.float32)
    for j in range(M):
        B[g.choice(K, 3, replace=False), j] = g.standard_normal(3)
    ref = A.astype(np.float64) @ B.astype(np.float64)
    size = np.abs(A).astype(np.float64) @ np.abs(B).astype(np.float64)
    assert np.max(np.abs(_product(fmm, A, B, tile, 0) - ref) / size) <= FORMS[tile][2] + 3 * ADDS


@pytest.mark.parametrize("tile", [512, 256])
def test_integers_through_a_permutation(fmm, tile):
    g, (bits_a, bits_b) = np.random.default_rng(10), FORMS[tile][3:]
    P = np.eye(K, dtype=np.float32)[g.permutation(K)]
    A = g.integers(-2 ** bits_a + 1, 2 ** bits_a, (M, K)).astype(np.float32)
    B = g.integers(-2 ** bits_b + 1, 2 ** bits_b, (K, M)).astype(np.float32)
    assert np.array_equal(_product(fmm, A, P, tile, 0), A @ P)
    assert np.array_equal(_product(fmm, P, B, tile, 0), P @ B)
