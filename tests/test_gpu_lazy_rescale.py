"""Eliminations of tiles whose pivots leave the range in which no step rescales.

L has few-bit entries and power-of-two diagonals down to 2^-20, so L L^T and every
intermediate of the elimination are exact in FP64 and only the square roots and the final
multiplications round: a few units in the last place of max|L|, whatever the pivots.
Pivots of 2^-40 drive the accumulated scale below 2^-64 within three steps, pivots near
2 above 2^64 within eight.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [16, 33, 100, 2064])
@pytest.mark.parametrize("small", [0.0, 0.5, 1.0])
def test_factor_of_exact_products(n, small):
    from paper_2201_00241_gb300 import rh
    rng = np.random.default_rng(n)
    L = np.tril(rng.integers(-1, 2, (n, n)) * 0.5, -1)
    L[np.abs(np.subtract.outer(np.arange(n), np.arange(n))) > 6] = 0.0     # few terms: 45 bits hold every sum
    np.fill_diagonal(L, np.where(rng.random(n) < small, 2.0 ** -20, 1.0))
    H = L @ L.T
    A = torch.from_numpy(np.ascontiguousarray(H.T)).cuda().t()
    info = rh.potrf(A)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert np.abs(np.tril(A.cpu().numpy()) - L).max() <= 16 * np.finfo(float).eps
