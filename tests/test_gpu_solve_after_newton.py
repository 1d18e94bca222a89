"""rh_solve on the factors that a power flow leaves: those of its last Newton step.

One Newton step from x0 (the single and the batched power flow), after an adjoint at another
point of the same grid and on a grid that has factored nothing else: the step's factors are
those of J_x(x0), so both solves match the oracle's at x0 to 1e-10 of the largest entry (the
solves' tolerance elsewhere).  Shapes: tails factored in one CTA and tile by tile, a grid
that is all tail, and a tail whose triangle does not fit in shared memory beside x.  A solve
captured before the power flow and replayed after it solves with the new factors too.
"""
import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPES = [((5, 6, 2, 1), 0), ((118, 186, 54, 20220100), 0), ((700, 1100, 100, 12), 80), ((700, 1100, 100, 12), 512)]


def near(a, b):
    return np.abs(a - b).max() <= 1e-10 * np.abs(b).max()


@pytest.mark.parametrize("shape,max_tail", SHAPES)
@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("adjoint_before", [False, True])
def test_solves_use_the_last_newton_step(shape, max_tail, batch, adjoint_before):
    from paper_2201_00241_gb300 import rh
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0, max_tail=max_tail), OracleGrid(g)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    rng = np.random.default_rng(3)
    R = np.asfortranarray(rng.normal(size=(lg.n_x, 3)))
    if adjoint_before:
        lg.powerflow(st.x)
        lg.adjoint()
        assert near(lg.solve(R), o.solve(so.x, so.p, R))
    x0 = st.x + 0.02 * rng.normal(size=lg.n_x)
    if batch:
        rh.batch_powerflow([lg], [x0], max_iter=1)
    else:
        assert lg.powerflow(x0, max_iter=1, raise_on_noconv=False)[1] == 1
    for trans in (False, True, False):
        assert near(lg.solve(R, trans=trans), o.solve(x0, so.p, R, trans=trans))
    lg.powerflow(st.x)
    lg.adjoint()
    for trans in (False, True):
        assert near(lg.solve(R, trans=trans), o.solve(so.x, so.p, R, trans=trans))


@pytest.mark.parametrize("shape,max_tail", SHAPES)
def test_captured_solve_follows_the_factors(shape, max_tail):
    from paper_2201_00241_gb300 import rh
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0, max_tail=max_tail), OracleGrid(g)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    lg.powerflow(st.x)
    lg.adjoint()
    rng = np.random.default_rng(4)
    R = rng.normal(size=(2, lg.n_x))
    Rd, lib = torch.from_numpy(R).cuda(), rh.load()
    lg.solve(R.T)                                   # the workspace exists before the capture
    s, cg = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s), torch.cuda.graph(cg, stream=s):
        rh._check(lib.rh_solve(lg._h, rh._ptr(Rd), lg.n_x, 2, 1, rh.C.c_void_p(s.cuda_stream), rh.RH_DEVICE_PTRS))
    x0 = st.x + 0.02 * rng.normal(size=lg.n_x)
    lg.powerflow(x0, max_iter=1, raise_on_noconv=False)
    for x in (x0, st.x):
        Rd.copy_(torch.from_numpy(R))
        cg.replay()
        torch.cuda.synchronize()
        assert near(Rd.cpu().numpy().T, o.solve(x, so.p, R.T, trans=True))
        lg.powerflow(st.x)
        lg.adjoint()
