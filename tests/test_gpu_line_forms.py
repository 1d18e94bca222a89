"""The line schedules where the dense tail is swept level by level, and the line between the
kernels of few and of many directions.

A tail whose triangle does not fit in shared memory beside x (max_tail 512) leaves the single
solves, the products of few directions and the batched form of those with schedules over
every level, in CTAs of 256 threads (up to 1024 rows of x) and of 512.  Newton, the adjoint,
both solves and products of one direction, of as many as two an SM, and of one more, match
the oracle to 1e-10 of the largest entry, the products' tolerance elsewhere.
"""
import numpy as np
import pytest

from oracle import OracleGrid
from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def near(a, b):
    return np.abs(a - b).max() <= 1e-10 * np.abs(b).max()


@pytest.mark.parametrize("shape,max_tail,rows", [((450, 700, 60, 7), 512, (513, 1024)), ((700, 1100, 100, 12), 512, (1025, 9999)),
                                                 ((450, 700, 60, 7), 0, (513, 1024)), ((700, 1100, 100, 12), 0, (1025, 9999))])
def test_swept_tails_and_both_sides_of_two_directions_an_sm(shape, max_tail, rows):
    from paper_2201_00241_gb300 import rh
    slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0, max_tail=max_tail), OracleGrid(g)
    assert rows[0] <= lg.n_x <= rows[1] and (lg.dims.tail_vars > 500) == (max_tail == 512)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    x, _, res, _ = lg.powerflow(None, tol=1e-12)
    assert res <= 1e-12 and np.abs(x - so.x).max() <= 1e-8
    lg.powerflow(st.x)
    lam, grad, F = lg.adjoint()
    lo, go, Fo = o.adjoint(so.x, so.p, so.pd, so.qd)
    assert near(lam, lo) and near(grad, go) and F == pytest.approx(Fo, rel=1e-12)
    R = np.random.default_rng(2).normal(size=(lg.n_x, 2))
    for trans in (False, True):
        assert near(lg.solve(R, trans=trans), o.solve(so.x, so.p, R, trans=trans))
    H = o.hessvec(so.x, so.p, so.pd, so.qd, np.eye(lg.n_p))
    assert near(lg.reduced_hessian()[0], H)
    items, refs = [], []
    for n in (1, slots, slots + 1):
        W = gg.random_directions(lg.n_p, n, n)
        assert near(lg.hessvec(W), H @ W)
        Wd = torch.from_numpy(np.ascontiguousarray(W.T)).cuda().t()
        items.append((lg, Wd, torch.empty_like(Wd), torch.empty(rh.work_doubles(lg, n), dtype=torch.float64, device="cuda")))
        refs.append(H @ W)
    for batch in (items[:1], items):
        rh.batch_hessvec(batch, 0)
        torch.cuda.synchronize()
        for (_, _, HW, _), ref in zip(batch, refs):
            assert near(HW.cpu().numpy(), ref)
            HW.zero_()
