"""Index checks on the GPU where launches take other kernels by width and size.

The index-checking build (librh_bounds.so) in a child process: products and full Hessians of
more directions than two an SM (several directions per CTA, the reach-restricted sweeps, the
folded first level) and of fewer (one per CTA, x in shared memory), on both CTA shapes, with
a tail solved in shared memory and one swept like the rest, batched launches with one
direction per CTA beside the others, and solves on a Newton step's factors.  The error word
stays 0 and the results match the oracle to the products' 1e-10 of the largest entry.
"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys, ctypes as C
import numpy as np
sys.path.insert(0, ROOT)
from paper_2201_00241_gb300 import build as B
B.LIB = B.build(bounds=True)
import torch
from paper_2201_00241_gb300 import rh, gridgen as gg
from oracle import OracleGrid

lib, en, err = rh.load(), C.c_int32(0), C.c_uint32(0)
slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count
out, grids = {}, {}
rel = lambda a, b: float(np.abs(a - b).max() / np.abs(b).max())

def item(lg, n):
    W = torch.from_numpy(np.ascontiguousarray(gg.random_directions(lg.n_p, n, n).T)).cuda().t()
    return (lg, W, torch.empty((n, lg.n_p), dtype=torch.float64, device="cuda").t(),
            torch.empty(rh.work_doubles(lg, n), dtype=torch.float64, device="cuda"))

for name, shape, tail in [("wide", (slots + 100, slots + 260, slots // 2 + 20, 3), 0), ("large", (700, 1100, 100, 12), 0),
                          ("swept", (700, 1100, 100, 12), 512), ("small", (118, 186, 54, 20220100), 0)]:
    g = gg.make_grid(*shape)
    lg, o = rh.Grid(g, device=0, max_tail=tail), OracleGrid(g)
    st, so = lg.plant(), o.plant()
    lg.set_state(st.p, st.pd, st.qd)
    assert (lg.n_p > slots) == (name == "wide") and (lg.n_x > 1024) == (name in ("large", "swept"))
    rng = np.random.default_rng(1)
    R, x0, worst = rng.normal(size=(lg.n_x, 3)), st.x + 0.02 * rng.normal(size=lg.n_x), 0.0
    for batch in (True, False):
        if batch:
            rh.batch_powerflow([lg], [x0], max_iter=1)
        else:
            lg.powerflow(x0, max_iter=1, raise_on_noconv=False)
        for trans in (False, True):
            worst = max(worst, rel(lg.solve(R, trans=trans), o.solve(x0, so.p, R, trans=trans)))
    lg.powerflow(st.x)
    H, _, _ = lg.reduced_hessian()
    Ho = o.hessvec(so.x, so.p, so.pd, so.qd, np.eye(lg.n_p))
    worst = max(worst, rel(H, Ho))
    lg.adjoint()
    worst = max(worst, rel(lg.hessian(), Ho), rel(lg.hessian(block_n=100, concurrent=False), Ho))
    for N in (1, 152, slots, slots + 1, 3 * slots):
        W = gg.random_directions(lg.n_p, N, N)
        worst = max(worst, rel(lg.hessvec(W), Ho @ W))
    grids[name] = (lg, Ho)
    out[name] = worst
for mix in ([("large", 3), ("small", 40), ("swept", 9)], [("large", 170), ("wide", 5), ("small", 300), ("swept", 2)]):
    items = [item(grids[n][0], k) for n, k in mix]
    for width in (0, 3):
        rh.batch_hessvec(items, width)
        torch.cuda.synchronize()
        for (n, _), (_, W, HW, _) in zip(mix, items):
            out[n] = max(out[n], rel(HW.cpu().numpy(), grids[n][1] @ W.cpu().numpy()))
assert lib.rh_bounds_check(0, C.byref(en), C.byref(err)) == 0
print(json.dumps({"enabled": en.value, "errors": err.value, "worst": out}))
"""


def test_no_index_outside_its_array_at_any_width():
    r = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT", repr(ROOT))], capture_output=True, text=True,
                       cwd=ROOT, timeout=1200)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert res["enabled"] == 1 and res["errors"] == 0, res
    assert max(res["worst"].values()) <= 1e-10, res
