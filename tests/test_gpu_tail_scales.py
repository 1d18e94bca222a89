"""The dense tail's elimination with pivots far from 1.

Every impedance divided by 2^k multiplies J_x by 2^k exactly, so the factors and both solves
keep their digits and only exponents move: the solutions equal those of k = 0 times 2^-k, bit
for bit, however often a step rescales.  k = -20 and 20 drive the accumulated scale beyond
2^64 within three or four pivots, k = 80 and -80 put every pivot there.  Tails in one CTA
(a partial tile, three tiles) and tile by tile.
"""
import dataclasses

import numpy as np
import pytest

from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,max_tail", [((90, 150, 20, 5), 0), ((700, 1100, 100, 12), 48), ((700, 1100, 100, 12), 100)])
def test_scaled_networks_keep_every_digit(shape, max_tail):
    from paper_2201_00241_gb300 import rh
    g0, sols = gg.make_grid(*shape), {}
    for k in (0, -80, -20, 20, 80):
        f = 2.0 ** -k
        lg = rh.Grid(dataclasses.replace(g0, r=g0.r * f, x=g0.x * f, b=g0.b / f), device=0, max_tail=max_tail)
        st = lg.plant()
        lg.set_state(st.p, st.pd, st.qd)
        lg.powerflow(st.x, max_iter=0, raise_on_noconv=False)
        lg.refactor()
        R = np.random.default_rng(5).normal(size=(lg.n_x, 2))
        sols[k] = [lg.solve(R, trans=t) / f for t in (False, True)]
    for k, s in sols.items():
        for got, ref in zip(s, sols[0]):
            assert np.isfinite(got).all() and np.array_equal(got, ref), k
