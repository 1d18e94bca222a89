"""Batched launches whose largest grids run one direction per CTA beside the other items.

All items on large grids, large and small ones mixed, blocks of one direction, an empty
item, item-owned workspaces, more items than one launch holds, and the launch replayed from
a CUDA graph.  Every item's HW is the single call's up to the order of summation: 1e-10 of
max|HW|, the tolerance of the product tests.
"""
import numpy as np
import pytest

from paper_2201_00241_gb300 import gridgen as gg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def nets():
    from paper_2201_00241_gb300 import rh
    out = {}
    for name, shape in dict(s=(118, 186, 54, 1), m=(540, 800, 60, 11), l=(700, 1100, 100, 12), x=(1600, 2500, 300, 5)).items():
        lg = rh.Grid(gg.make_grid(*shape), device=0)
        st = lg.plant()
        lg.set_state(st.p, st.pd, st.qd)
        lg.powerflow(st.x)
        lg.adjoint()
        out[name] = lg
    return out


@pytest.mark.parametrize("mix", [[("l", 1)], [("x", 5), ("l", 40)], [("s", 30), ("x", 160), ("m", 7), ("s", 1), ("l", 3)],
                                 [("s", 200), ("x", 0), ("x", 9)], [("s", 2)] * 20 + [("x", 4)] + [("s", 3)] * 20 + [("l", 2)]],
                         ids=["one", "large", "mixed", "empty", "two_launches"])
@pytest.mark.parametrize("graph", [False, True])
def test_batch_matches_single_calls(nets, mix, graph):
    from paper_2201_00241_gb300 import rh
    items, refs = [], []
    for k, (name, n) in enumerate(mix):
        lg = nets[name]
        W = torch.from_numpy(np.ascontiguousarray(gg.random_directions(lg.n_p, max(n, 1), k).T[:n])).cuda().t()
        HW = torch.full((n, lg.n_p), float("nan"), dtype=torch.float64, device="cuda").t()
        items.append((lg, W, HW, torch.empty(max(1, rh.work_doubles(lg, n)), dtype=torch.float64, device="cuda")))
        refs.append(lg.hessvec(W.cpu().numpy()) if n else None)
    if graph:
        s, cg = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.stream(s), torch.cuda.graph(cg, stream=s):
            rh.batch_hessvec(items, 0, stream=rh.C.c_void_p(s.cuda_stream))
        cg.replay()
    else:
        rh.batch_hessvec(items, 0)
    torch.cuda.synchronize()
    for (lg, W, HW, _), ref in zip(items, refs):
        if ref is not None:
            assert np.abs(HW.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
