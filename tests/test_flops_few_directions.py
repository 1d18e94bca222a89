"""rh_reduced_hessian_flops where the launches run one direction per CTA (n_p up to 2 n_sm).

Every sweep then covers all rows: the count follows from the exported L and U patterns alone,
with the dense tail as a full triangle, or, where that triangle does not fit in shared memory
beside x, sparse like the rest.  One direction more than 2 n_sm brings the reach back.
"""
import ctypes as C

import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg
from paper_2201_00241_gb300 import rh


@pytest.mark.parametrize("shape,max_tail,dense", [((30, 41, 6, 4), 0, True), ((118, 186, 54, 20220100), 0, True),
                                                  ((700, 1100, 100, 12), 0, True), ((700, 1100, 100, 12), 512, False)])
def test_counts_every_row(shape, max_tail, dense):
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=-1, max_tail=max_tail), OracleGrid(g)
    d, sym = lg.dims, lg.symbolic()
    nx, n_p, T = d.n_x, d.n_p, d.tail_vars
    row = np.repeat(np.arange(nx), np.diff(sym["Lp"]))
    in_tail = int(((row >= nx - T) & (sym["Lj"] >= nx - T)).sum())
    lower = d.nnz_l - (in_tail - T * (T - 1) // 2 if dense else 0)          # FMAs of a sweep
    pairs = {(min(a, b), max(a, b)) for a, b in zip(g.fr, g.to)}
    ref = int(np.flatnonzero(g.bus_type == 0)[0])
    deg = sum(ref in p for p in pairs)
    st = o.plant()
    nnz_jp = o.jacobians_csc(st.x, st.p)[1].nnz
    proj = 6 * g.n_bus + 16 * len(pairs) + 4 * (1 + deg) + 2 * (1 + 2 * deg) + 1 + int((g.bus_type == 1).sum())
    want = n_p * (proj + 2 * (4 * lower + nnz_jp))
    lib, a, e = rh.load(), C.c_double(), C.c_double()
    for n_sm, all_rows in ((-(-n_p // 2), True), (max(152, n_p), True), ((n_p - 1) // 2, False)):
        assert lib.rh_reduced_hessian_flops(lg._h, n_sm, C.byref(a), C.byref(e)) == 0
        assert (e.value == want) if all_rows else (e.value < want or T == nx or not dense)
