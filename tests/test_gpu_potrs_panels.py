"""Cholesky solves with few right-hand sides, one launch per panel of 96 columns.

Sizes at the edges of the panels and of their 16-row blocks, strips of 8 and of 32
rows, one and several right-hand sides, and calls on both sides of the rule's lines (more
than 128 rows, at most 16 right-hand sides, at most 16384 numbers).  Two solves of one system in different summation orders
differ by about n eps cond(A) relative to max|x|; the test allows 8 n eps cond(A).
"""
import numpy as np
import pytest

from oracle import cholesky, cholesky_solve

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
EPS = np.finfo(float).eps


@pytest.mark.parametrize("n,nrhs", [(96, 1), (128, 2), (129, 1), (145, 16), (191, 2), (192, 1), (193, 17),
                                    (290, 3), (577, 1), (1019, 3), (1024, 16), (1300, 13)])
def test_panel_solves_match_oracle(n, nrhs):
    from paper_2201_00241_gb300 import rh
    rng = np.random.default_rng(100 * n + nrhs)
    A = rng.standard_normal((n, n))
    H = A @ A.T / n + np.eye(n)
    L, info = cholesky(H)
    assert info == 0
    B = rng.standard_normal((n, nrhs))
    ref = cholesky_solve(L, B)
    Ld = torch.from_numpy(np.ascontiguousarray(np.tril(L).T + np.tril(np.full((n, n), np.nan), -1))).cuda().t()
    buf = torch.full((nrhs, n + 3), 7.0, dtype=torch.float64, device="cuda")
    buf[:, :n] = torch.from_numpy(np.ascontiguousarray(B.T))
    X = buf.t()[:n, :]
    rh.potrs(Ld, X)
    torch.cuda.synchronize()
    assert np.abs(X.cpu().numpy() - ref).max() <= 8 * n * EPS * np.linalg.cond(H) * np.abs(ref).max()
    assert bool((buf[:, n:] == 7.0).all())              # rows beyond n untouched; the NaN above L's diagonal unread
