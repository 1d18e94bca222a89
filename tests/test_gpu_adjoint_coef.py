"""The kernels behind rh_adjoint's outputs other than the solve, on both of their forms.

A network whose largest bus has at most 32 admittance entries runs one entry per lane; a
star of 40 branches runs one bus per thread.  grad F, F and H (through the projection's
coefficients) are the oracle's to 1e-10 of their largest entry, the tolerance of the
existing parity tests; the slack is a leaf, a hub, and an ordinary bus.
"""
import dataclasses

import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def star(n, seed):
    """make_grid's network with every branch's far end moved so that bus 0 is a hub of n - 1 neighbours."""
    g = gg.make_grid(n, n - 1, max(1, n // 4), seed)
    return dataclasses.replace(g, fr=np.zeros(n - 1, np.int32), to=np.arange(1, n, dtype=np.int32))


@pytest.mark.parametrize("make", [lambda: star(41, 3), lambda: star(30, 5), lambda: gg.make_grid(2, 1, 1, 3),
                                  lambda: gg.make_grid(400, 640, 80, 7)], ids=["hub40", "hub29", "two", "mesh"])
def test_adjoint_outputs_match_oracle(make):
    from paper_2201_00241_gb300 import rh
    g = make()
    lg, o = rh.Grid(g, device=0), OracleGrid(g)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    lg.powerflow(st.x)
    lam, grad, F = lg.adjoint()
    lam_o, grad_o, F_o = o.adjoint(so.x, so.p, so.pd, so.qd)
    H = o.hessvec(so.x, so.p, so.pd, so.qd, np.eye(lg.n_p))
    assert np.abs(lam - lam_o).max() <= 1e-10 * np.abs(lam_o).max()
    assert np.abs(grad - grad_o).max() <= 1e-10 * np.abs(grad_o).max()
    assert F == pytest.approx(F_o, rel=1e-12)
    assert np.abs(lg.hessvec(np.eye(lg.n_p)) - H).max() <= 1e-10 * np.abs(H).max()
