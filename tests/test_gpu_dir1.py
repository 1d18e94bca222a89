"""Products of few directions: one direction per CTA, x in shared memory (k_dir1).

Networks below and above the line between the two CTA shapes (1024 rows of x), with buses
of one row (every bus a generator) and of two, with and without a dense tail; blocks of
one direction and of several, identity columns, and the reduced Hessian in two launches.
The projection and both solves are the oracle's operations in another order, so the
tolerance is the one every product is held to: 1e-10 of max|HW|.
"""
import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL_HW = 1e-10


@pytest.mark.parametrize("shape", [(2, 1, 1, 3), (3, 2, 3, 5), (30, 41, 6, 4), (61, 90, 61, 8), (118, 186, 54, 20220100),
                                   (540, 800, 60, 11), (700, 1100, 100, 12)])
def test_few_directions_match_oracle(shape):
    from paper_2201_00241_gb300 import rh
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0), OracleGrid(g)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    lg.powerflow(st.x)
    H2, _, _ = lg.reduced_hessian()
    lg.adjoint()
    H = o.hessvec(so.x, so.p, so.pd, so.qd, np.eye(lg.n_p))
    top = np.abs(H).max()
    assert np.abs(H2 - H).max() <= TOL_HW * top
    for N in (1, 3, 17):
        W = gg.random_directions(lg.n_p, N, N)
        ref = o.hessvec(so.x, so.p, so.pd, so.qd, W)
        assert np.abs(lg.hessvec(W) - ref).max() <= TOL_HW * max(np.abs(ref).max(), 1e-300)
    assert np.abs(lg.hessian(block_n=5) - H).max() <= TOL_HW * top
    k = lg.n_p // 2
    assert np.abs(lg.hessian_columns(k, lg.n_p - k) - H[:, k:]).max() <= TOL_HW * top
