"""Dense tails factored in one CTA beside the pivot steps (up to 64 variables).

Tails of one partial tile, of full tiles and of a partial last tile, the largest that takes
this path, and the first that does not; grids whose every variable is in the tail.  Both
solves on the factors match the oracle's to 1e-10 of the largest entry and a power flow
from a flat start reaches the oracle's state (its triangles are the Newton step's): the
tolerances of the existing parity tests.
"""
import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,max_tail,tail", [((2, 1, 1, 3), 0, 2), ((5, 6, 2, 1), 0, 7), ((90, 150, 20, 5), 0, 15),
                                                 ((118, 186, 54, 20220100), 0, 16),
                                                 ((118, 186, 54, 20220100), 31, None),
                                                 ((118, 186, 54, 20220100), 48, None),
                                                 ((700, 1100, 100, 12), 64, None), ((700, 1100, 100, 12), 61, None),
                                                 ((700, 1100, 100, 12), 80, None)])
def test_solves_and_power_flow_match_oracle(shape, max_tail, tail):
    from paper_2201_00241_gb300 import rh
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0, max_tail=max_tail), OracleGrid(g)
    if tail is not None:
        assert lg.dims.tail_vars == tail
    else:
        assert max_tail - 2 < lg.dims.tail_vars <= max_tail
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    x, _, res, _ = lg.powerflow(None, tol=1e-12)
    assert res <= 1e-12 and np.abs(x - so.x).max() <= 1e-8
    lg.powerflow(st.x)
    lg.adjoint()
    R = np.asfortranarray(np.random.default_rng(7).normal(size=(lg.n_x, 3)))
    for trans in (False, True):
        ref = o.solve(so.x, so.p, R, trans=trans)
        got = lg.solve(R, trans=trans)
        assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()
