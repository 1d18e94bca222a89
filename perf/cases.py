"""What a program built on this package has it do, as cases with inputs, one pass and a plain 64-bit reference.

A case is a call pattern (``kind``) on a grid shape (buses, branches, generators) with a width N:

* ``hessvec``      a block of N directions through ``Grid.hessvec`` (an optimiser's products, N = 1 in a CG loop)
* ``hessian``      one operating point's Jacobians, factors, adjoint and full reduced Hessian in one call
* ``adjoint``      one operating point's factors, lambda and reduced gradient (first-order methods)
* ``solve``        batched solves with J_x or its transpose on host buffers (sensitivities, both directions)
* ``batch``        several (grid, W) items of one launch: load scenarios, or requests on grids of different sizes
* ``resolve``      Newton power flow of several load scenarios of one network
* ``track``        a tracking update: new loads, warm power flow, adjoint, Hessian, Cholesky and step
* ``newton_cg``    F, its gradient and a product through the autograd Function at two successive points
* ``cholesky``     the dense factorisation and solve on their own

The shapes are those of the repository's generator and tests.  The operating point is planted: smooth voltages
drawn from the seed, and the loads and generations that make them a solution, formed here with numpy.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2201_00241_gb300 import autograd, gridgen, rh


def listed():
    return [
        # one product on a small network: an optimiser's inner loop, where latency and launches count
        dict(name="product_118_n1", kind="hessvec", buses=118, branches=186, gens=54, n=1, grid_seed=20220100),
        # the small network's whole second-order model at one operating point
        dict(name="hessian_118", kind="hessian", buses=118, branches=186, gens=54, n=107, grid_seed=20220100),
        # a truncated-Newton step through torch.autograd on a mid-size network: F, gradient, product, twice
        dict(name="newton_cg_1354", kind="newton_cg", buses=1354, branches=1991, gens=260, n=1, grid_seed=20220101),
        # eight load scenarios of one network: their power flows, and 64 directions on each in one launch
        dict(name="resolve_1354_x8", kind="resolve", buses=1354, branches=1991, gens=260, n=8, grid_seed=20220101),
        dict(name="scenarios_1354_8x64", kind="batch", buses=1354, branches=1991, gens=260, n=64, items=8, mixed=False,
             grid_seed=20220101),
        # a tracking controller's update
        dict(name="track_1354", kind="track", buses=1354, branches=1991, gens=260, n=519, grid_seed=20220101),
        # odd width on the next shape: directions that fill neither the CTAs nor the warps evenly
        dict(name="products_2869_n45", kind="hessvec", buses=2869, branches=4582, gens=510, n=45, grid_seed=20220104),
        # a serving round: requests of uneven widths on networks of four sizes in one launch
        dict(name="serving_round", kind="batch", buses=9241, branches=16049, gens=1445, n=128, items=15, mixed=True,
             grid_seed=20220102),
        # the largest shape: first-order set-up, a block of directions, and the full reduced Hessian
        dict(name="adjoint_9241", kind="adjoint", buses=9241, branches=16049, gens=1445, n=1, grid_seed=20220102),
        dict(name="products_9241_n256", kind="hessvec", buses=9241, branches=16049, gens=1445, n=256,
             grid_seed=20220102),
        dict(name="hessian_9241", kind="hessian", buses=9241, branches=16049, gens=1445, n=2889, grid_seed=20220102),
        # the dense factorisation at the order of a mid-size network's Hessian
        dict(name="cholesky_1019", kind="cholesky", order=1019, n=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hessvec", "hessvec", "hessvec", "hessian", "hessian", "adjoint", "solve", "batch", "batch",
                       "resolve", "track", "newton_cg", "cholesky"])
    if kind == "cholesky":
        return dict(kind=kind, order=_log(rng, 107, 2400), n=rng.randint(1, 16))
    buses = _log(rng, 118, 1500 if kind in ("newton_cg", "resolve") else 4600)
    branches = int(buses * rng.uniform(1.45, 1.72))
    gens = max(3, int(buses * rng.uniform(0.15, 0.45)))
    case = dict(kind=kind, buses=buses, branches=branches, gens=gens, grid_seed=rng.randrange(1, 1 << 30))
    if kind == "hessvec":
        case["n"] = _log(rng, 1, 256)
    elif kind == "solve":
        case.update(n=_log(rng, 1, 96), trans=bool(rng.randrange(2)))
    elif kind == "batch":
        case.update(n=_log(rng, 2, 128), items=rng.randint(2, 15), mixed=bool(rng.randrange(2)))
    elif kind == "resolve":
        case["n"] = rng.randint(1, 16)
    elif kind in ("hessian", "track"):
        if kind == "track":       # Cholesky wants a convex point: the shapes whose costs give one
            case.update(rng.choice([dict(buses=118, branches=186, gens=54, grid_seed=20220100),
                                    dict(buses=1354, branches=1991, gens=260, grid_seed=20220101),
                                    dict(buses=2869, branches=4582, gens=510, grid_seed=20220104)]))
            case["load"] = rng.uniform(0.97, 1.03)
        case["n"] = 2 * case["gens"] - 1
    else:
        case["n"] = 1
    return case


# ---- inputs -------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=16)
def _record(buses, branches, gens, seed):
    return gridgen.make_grid(buses, branches, gens, seed)


def _shapes(case):
    """(buses, branches, gens, grid seed) of the case's network, and of each item of a mixed batch."""
    own = (case["buses"], case["branches"], case["gens"], case["grid_seed"])
    if not case.get("mixed"):
        return [own] * case.get("items", 1)
    small = [(118, 186, 54, 20220100)] * 8 + [(1354, 1991, 260, 20220101)] * 4 + [(2869, 4582, 510, 20220104)] * 2
    pick = (small + [own])[-case["items"]:]
    return pick


class _Net:
    """Admittances and index maps of one grid record (x: angles at PV then PQ buses, magnitudes at PQ buses;
    p: magnitudes at generator buses, generations at PV buses)."""

    def __init__(self, g):
        self.g, n = g, g.n_bus
        y = 1.0 / (g.r + 1j * g.x)
        i = np.concatenate([g.fr, g.to, g.fr, g.to])
        j = np.concatenate([g.to, g.fr, g.fr, g.to])
        v = np.concatenate([-y, -y, y + 0.5j * g.b, y + 0.5j * g.b])
        key, at = np.unique(i.astype(np.int64) * n + j, return_inverse=True)
        self.i, self.j = key // n, key % n
        self.y = np.bincount(at, v.real, len(key)) + 1j * np.bincount(at, v.imag, len(key))
        t = g.bus_type
        self.ref = int(np.flatnonzero(t == 0)[0])
        self.pv, self.pq, self.gen = np.flatnonzero(t == 1), np.flatnonzero(t == 2), np.flatnonzero(t != 2)
        self.ang = np.concatenate([self.pv, self.pq])
        self.n_x, self.n_p = len(self.ang) + len(self.pq), len(self.gen) + len(self.pv)

    def injections(self, vm, va):
        v = vm * np.exp(1j * va)
        w = self.y * v[self.j]
        s = v * np.conj(np.bincount(self.i, w.real, len(vm)) + 1j * np.bincount(self.i, w.imag, len(vm)))
        return s.real, s.imag

    def smooth(self, rng):
        """A per-bus field of unit spread that varies slowly over the network."""
        n = self.g.n_bus
        f, deg = rng.standard_normal(n), np.bincount(self.i, minlength=n)
        for _ in range(30):
            f = np.bincount(self.i, f[self.j], n) / deg
        f -= f.mean()
        return f / f.std()

    def point(self, rng):
        """A planted operating point: (vm, va, x, p, pd, qd)."""
        g = self.g
        vm = np.clip(g.v_star + 0.01 * self.smooth(rng), 0.94, 1.06)
        va = g.theta_star + 0.02 * self.smooth(rng)
        va -= va[self.ref]
        P, Q = self.injections(vm, va)
        pd, qd = np.zeros(g.n_bus), np.zeros(g.n_bus)
        pd[self.pq], qd[self.pq] = -P[self.pq], -Q[self.pq]
        return vm, va, np.concatenate([va[self.ang], vm[self.pq]]), np.concatenate([vm[self.gen], P[self.pv]]), pd, qd


@functools.lru_cache(maxsize=16)
def _net(*shape):
    return _Net(_record(*shape))


def _unit(rng, rows, cols):
    w = rng.standard_normal((cols, rows))
    return (w / np.linalg.norm(w, axis=1, keepdims=True)).T      # column-major


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a.T)).cuda().t()


def _inputs(case, seed):
    """Everything that the seed decides, as numpy arrays."""
    rng = np.random.Generator(np.random.PCG64([seed, 7]))
    kind = case["kind"]
    if kind == "cholesky":
        n = case["order"]
        f = rng.standard_normal((n, 24))
        diag = rng.uniform(1.0, 30.0, n)
        return dict(f=f, diag=diag, b=rng.standard_normal((n, case["n"])))
    nets = [_net(*s) for s in _shapes(case)]
    first = nets[0]
    if kind == "batch":
        top = case["n"]
        widths = [top] * len(nets)
        if case["mixed"]:            # uneven widths of mean n, the same for every seed
            even = np.random.Generator(np.random.PCG64(case["grid_seed"])).integers(1, 2 * top, len(nets))
            widths = [max(1, int(w * top * len(nets) // even.sum())) for w in even]
        pts = [net.point(rng) for net in nets]
        return dict(nets=nets, points=pts, w=[_unit(rng, net.n_p, k) for net, k in zip(nets, widths)])
    pt = first.point(rng)
    d = dict(nets=nets, points=[pt])
    if kind in ("hessvec", "newton_cg"):
        d["w"] = _unit(rng, first.n_p, case["n"])
    if kind == "newton_cg":
        step = np.zeros(first.n_p)
        step[:len(first.gen)] = 0.002 * rng.standard_normal(len(first.gen))
        d["p1"] = pt[3] + step
    if kind == "solve":
        d["r"] = np.asfortranarray(rng.standard_normal((first.n_x, case["n"])))
    if kind == "resolve":
        d["scales"] = rng.uniform(0.96, 1.04, (case["n"], first.g.n_bus))
    if kind == "track":
        d["scales"] = case.get("load", 1.0 + 0.01 * rng.standard_normal()) * rng.uniform(0.98, 1.02, (1, first.g.n_bus))
    return d


def _ready(net, pt, adjoint=True):
    g = rh.Grid(net.g, device=0)
    g.set_state(pt[3], pt[4], pt[5])
    g.powerflow(pt[2], tol=1e-10)
    if adjoint:
        g.adjoint()
    return g


def prepare(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    if kind == "cholesky":
        f = torch.from_numpy(d["f"]).cuda()
        a = (f @ f.t() + torch.diag(torch.from_numpy(d["diag"]).cuda())).t()
        b = _dev(d["b"])
        return dict(kind=kind, a0=a, a=a.clone(), b0=b, b=_dev(d["b"]), work=torch.empty_like(b).reshape(-1))
    net, pt = d["nets"][0], d["points"][0]
    if kind == "hessvec":
        w = _dev(d["w"])
        return dict(kind=kind, grid=_ready(net, pt), w=w, hw=torch.empty_like(w))
    if kind == "hessian":
        return dict(kind=kind, grid=_ready(net, pt, False),
                    h=torch.empty((net.n_p, net.n_p), dtype=torch.float64, device="cuda").t())
    if kind == "adjoint":
        return dict(kind=kind, grid=_ready(net, pt, False))
    if kind == "solve":
        return dict(kind=kind, grid=_ready(net, pt), r=d["r"], trans=case["trans"])
    if kind == "batch":
        handles = {}          # requests on one network share its handle; scenarios have one each
        items = []
        for k, (n, p, w) in enumerate(zip(d["nets"], d["points"], d["w"])):
            key = id(n) if case["mixed"] else k
            if key not in handles:
                handles[key] = _ready(n, p)
            g, wd = handles[key], _dev(w)
            items.append((g, wd, torch.empty_like(wd),
                          torch.empty(rh.work_doubles(g, w.shape[1]), dtype=torch.float64, device="cuda")))
        return dict(kind=kind, items=items)
    if kind == "resolve":
        grids = []
        for s in d["scales"]:
            g = rh.Grid(net.g, device=0)
            g.set_state(pt[3], pt[4] * s, pt[5] * s)
            grids.append(g)
        return dict(kind=kind, grids=grids, x0=[pt[2]] * len(grids))
    if kind == "track":
        g = _ready(net, pt)
        s = d["scales"][0]
        return dict(kind=kind, grid=g, x0=pt[2], p=pt[3], pd=pt[4] * s, qd=pt[5] * s,
                    h=torch.empty((net.n_p, net.n_p), dtype=torch.float64, device="cuda").t())
    g = rh.Grid(net.g, device=0)
    g.set_state(pt[3], pt[4], pt[5])
    g.powerflow(pt[2], tol=1e-10)
    return dict(kind=kind, grid=g, v=torch.from_numpy(d["w"][:, 0].copy()).cuda(),
                ps=[torch.from_numpy(p).cuda().requires_grad_(True) for p in (pt[3], d["p1"])])


# ---- one pass -----------------------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "hessvec":
        return state["grid"].hessvec(state["w"], state["hw"])
    if kind == "hessian":
        return state["grid"].reduced_hessian(out=state["h"])
    if kind == "adjoint":
        return state["grid"].adjoint()
    if kind == "solve":
        return state["grid"].solve(state["r"], trans=state["trans"])
    if kind == "batch":
        rh.batch_hessvec(state["items"])
        return [hw for _, _, hw, _ in state["items"]]
    if kind == "resolve":
        return rh.batch_powerflow(state["grids"], state["x0"])[0]
    if kind == "track":
        g = state["grid"]
        g.set_state(state["p"], state["pd"], state["qd"])
        x = g.powerflow(state["x0"])[0]
        lam, grad, F = g.adjoint()
        d, p_next, L, info = g.rto_step(state["h"])
        return x, lam, grad, F, d, p_next, L, info
    if kind == "newton_cg":
        out = []
        for p in state["ps"]:
            F = autograd.reduced_objective(p, state["grid"])
            (grad,) = torch.autograd.grad(F, p, create_graph=True)
            (hv,) = torch.autograd.grad(grad, p, state["v"])
            out += [F.detach(), grad.detach(), hv]
        return out
    state["a"].copy_(state["a0"])
    state["b"].copy_(state["b0"])
    info = rh.potrf(state["a"])
    rh.potrs(state["a"], state["b"], state["work"])
    return state["a"], state["b"], info


# ---- what a pass cannot do without --------------------------------------------------------------------

@functools.lru_cache(maxsize=32)
def _counts(*shape):
    """Sizes of one network's sparse problem (symbolic phase only, no GPU)."""
    g = rh.Grid(_record(*shape), device=-1)
    d = g.dims
    c = dict(nx=d.n_x, np=d.n_p, jx=d.nnz_jx, jp=d.nnz_jp, lu=d.nnz_l + d.nnz_u, upd=d.refactor_updates,
             bus=d.n_bus, br=d.n_branch)
    g.close()
    return c


def _setup_work(c):
    """Jacobians, refactorisation, adjoint and gradient of one operating point: (bytes, flops)."""
    return 8 * (4 * c["bus"] + c["jx"] + c["nx"] + c["np"]), 2 * c["upd"] + 60 * c["br"] + 2 * (c["lu"] + c["jp"])


def _product_work(c, n):
    """n reduced-Hessian-vector products: factors and coefficients read once, W read and HW written once."""
    flops = n * (4 * c["jp"] + 4 * (c["lu"] - c["nx"]) + 16 * c["br"] + 8 * c["bus"])
    return 8 * (c["lu"] + c["jp"] + 8 * c["br"] + 2 * n * c["np"]), flops


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "cholesky":
        m = case["order"]
        return {"bytes": 8 * (m * m + 2 * m * n), "flops": m ** 3 / 3 + 2 * m * m * n}
    cs = [_counts(*s) for s in _shapes(case)]
    c = cs[0]
    if kind == "hessvec":
        b, f = _product_work(c, n)
    elif kind == "hessian":
        (b, f), (pb, pf) = _setup_work(c), _product_work(c, c["np"])
        b, f = b + pb - 8 * c["np"] ** 2, f + pf         # the identity is no input
    elif kind == "adjoint":
        b, f = _setup_work(c)
    elif kind == "solve":
        b, f = 8 * (c["lu"] + 2 * n * c["nx"]), 2 * n * c["lu"]
    elif kind == "batch":
        parts = [_product_work(q, n) for q in cs]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "resolve":
        b, f = n * 8 * (3 * c["bus"] + 2 * c["nx"]), n * 4 * (2 * c["upd"] + 60 * c["br"] + 2 * c["lu"])
    elif kind == "track":
        (sb, sf), (pb, pf) = _setup_work(c), _product_work(c, c["np"])
        b, f = sb + pb, 4 * sf + pf + c["np"] ** 3 / 3
    else:
        (sb, sf), (pb, pf) = _setup_work(c), _product_work(c, 1)
        b, f = 2 * (sb + pb), 2 * (4 * sf + pf)
    return {"bytes": b, "flops": f}


# ---- the same in plain 64 bits ------------------------------------------------------------------------

class _Dense:
    """The power-flow equations at one point, and their first and second derivatives, as dense matrices in the
    variables (angles of every bus, magnitudes of every bus)."""

    def __init__(self, net, vm, va, pd, device):
        self.net, n, t = net, net.g.n_bus, lambda a: torch.as_tensor(a, device=device)
        self.vm, self.va, self.pd, self.n, self.dev = t(vm), t(va), pd, n, device
        self.i, self.j = t(net.i), t(net.j)
        self.G, self.B = t(net.y.real.copy()), t(net.y.imag.copy())
        g = net.g
        self.ix = t(np.concatenate([net.ang, n + net.pq]))                 # x within (angles, magnitudes)
        self.iv = t(n + net.gen)                                          # the voltage part of p
        self.rows = t(np.concatenate([net.ang, n + net.pq]))               # equations within (P, Q)
        P, _ = net.injections(self.vm.cpu().numpy(), self.va.cpu().numpy())
        S = g.base_mva
        gen_mw = S * (P + pd)
        self.f1 = t(np.where(g.bus_type != 2, S * (2 * g.c2 * gen_mw + g.c1), 0.0))   # f' and f'' in per-unit power
        self.f2 = t(np.where(g.bus_type != 2, 2 * g.c2 * S * S, 0.0))
        self.F = float(np.sum((g.c2 * gen_mw ** 2 + g.c1 * gen_mw)[net.gen]))

    def jacobian(self):
        """d(P, Q)/d(angles, magnitudes), 2n x 2n."""
        n, i, j, vm = self.n, self.i, self.j, self.vm
        th = self.va[i] - self.va[j]
        c, s = torch.cos(th), torch.sin(th)
        a, b = self.G * c + self.B * s, self.G * s - self.B * c
        vi, vj = vm[i], vm[j]
        J = torch.zeros(2 * n, 2 * n, dtype=torch.float64, device=self.dev)
        off = i != j
        for row, val in ((i, a), (n + i, b)):
            J.index_put_((row, n + j), vi * val, accumulate=True)
            J.index_put_((row, n + i), vj * val, accumulate=True)
        for row, val in ((i, vi * vj * b), (n + i, -vi * vj * a)):
            val = torch.where(off, val, torch.zeros_like(val))
            J.index_put_((row, j), val, accumulate=True)
            J.index_put_((row, i), -val, accumulate=True)
        return J

    def hess_product(self, wp, wq, X):
        """(Hess of sum_i wp_i P_i + wq_i Q_i) X for the columns of X (rows: angles, magnitudes)."""
        n, i, j, vm = self.n, self.i, self.j, self.vm
        th = self.va[i] - self.va[j]
        c, s = torch.cos(th), torch.sin(th)
        A, C = wp[i] * self.G - wq[i] * self.B, wp[i] * self.B + wq[i] * self.G
        phi, dphi = A * c + C * s, C * c - A * s
        vi, vj = vm[i], vm[j]
        off = (i != j).double()
        idx = [i, j, n + i, n + j]
        m = {}
        m[0, 0] = m[1, 1] = -vi * vj * phi * off
        m[0, 1] = vi * vj * phi * off
        m[2, 3] = phi
        m[0, 2], m[1, 2] = vj * dphi * off, -vj * dphi * off
        m[0, 3], m[1, 3] = vi * dphi * off, -vi * dphi * off
        r, k, v = [], [], []
        for (p, q), val in m.items():
            r.append(idx[p]), k.append(idx[q]), v.append(val)
            if p != q:
                r.append(idx[q]), k.append(idx[p]), v.append(val)
        M = torch.sparse_coo_tensor(torch.stack([torch.cat(r), torch.cat(k)]), torch.cat(v), (2 * n, 2 * n))
        return torch.sparse.mm(M.coalesce(), X)


def _factored(D):
    J = D.jacobian()
    Jx = J[D.rows][:, D.ix].contiguous()
    Jv = J[D.rows][:, D.iv].contiguous()
    grad_ref = J[D.net.ref].clone()
    del J
    return Jx, Jv, grad_ref, torch.linalg.lu_factor(Jx)


def _solve(lu, Jx, R, trans=False):
    """One step of refinement on the dense factors."""
    A = Jx.t() if trans else Jx
    X = torch.linalg.lu_solve(*lu, R, adjoint=trans)
    return X + torch.linalg.lu_solve(*lu, R - A @ X, adjoint=trans)


def _first_order(D, fac):
    """(lambda, grad F): J_x^T lambda = -grad_x f, grad F = grad_p f + J_p^T lambda."""
    Jx, Jv, gr, lu = fac
    net = D.net
    c = D.f1[net.ref]
    lam = _solve(lu, Jx, -(c * gr[D.ix])[:, None], True)[:, 0]
    grad = torch.cat([c * gr[D.iv] + Jv.t() @ lam, D.f1[torch.as_tensor(net.pv, device=D.dev)] - lam[:len(net.pv)]])
    return lam, grad


def _second_order(D, fac, lam, W):
    """(Hess F) W for the columns of W."""
    Jx, Jv, gr, lu = fac
    net, n, k = D.net, D.n, W.shape[1]
    nv, npv, na = len(net.gen), len(net.pv), len(net.ang)
    R = Jv @ W[:nv]
    R[:npv] -= W[nv:]
    Z = -_solve(lu, Jx, R)
    del R
    X = torch.zeros(2 * n, k, dtype=torch.float64, device=D.dev)
    X[D.ix], X[D.iv] = Z, W[:nv]
    del Z
    wp, wq = torch.zeros(n, dtype=torch.float64, device=D.dev), torch.zeros(n, dtype=torch.float64, device=D.dev)
    wp[torch.as_tensor(net.ang, device=D.dev)] = lam[:na]
    wq[torch.as_tensor(net.pq, device=D.dev)] = lam[na:]
    wp[net.ref] += D.f1[net.ref]
    Y = D.hess_product(wp, wq, X) + D.f2[net.ref] * gr[:, None] * (gr @ X)[None, :]
    del X
    psi = -_solve(lu, Jx, Y[D.ix], True)
    return torch.cat([Y[D.iv] + Jv.t() @ psi, D.f2[torch.as_tensor(net.pv, device=D.dev)][:, None] * W[nv:] - psi[:npv]])


def _newton(net, vm, va, p, pd, qd, device, steps=8):
    vm, va = vm.copy(), va.copy()
    vm[net.gen] = p[:len(net.gen)]
    pg = np.zeros(net.g.n_bus)
    pg[net.pv] = p[len(net.gen):]
    for _ in range(steps):
        P, Q = net.injections(vm, va)
        res = np.concatenate([(P - pg + pd)[net.ang], (Q + qd)[net.pq]])
        D = _Dense(net, vm, va, pd, device)
        Jx, _, _, lu = _factored(D)
        dx = _solve(lu, Jx, torch.as_tensor(res, device=device)[:, None])[:, 0].cpu().numpy()
        va[net.ang] -= dx[:len(net.ang)]
        vm[net.pq] -= dx[len(net.ang):]
        if np.abs(dx).max() < 1e-13:
            break
    return vm, va, np.concatenate([va[net.ang], vm[net.pq]])


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind, d = case["kind"], _inputs(case, seed)
    if kind == "cholesky":
        f = torch.from_numpy(d["f"]).to(dev)
        a = f @ f.t() + torch.diag(torch.from_numpy(d["diag"]).to(dev))
        L = torch.linalg.cholesky(a)
        x = torch.cholesky_solve(torch.from_numpy(d["b"]).to(dev), L)
        return torch.tril(L) + torch.triu(a, 1), x, None
    net = d["nets"][0]
    if kind == "batch":
        out, cache = [], {}
        for k, (nt, pt, w) in enumerate(zip(d["nets"], d["points"], d["w"])):
            key = id(nt) if case["mixed"] else k
            if key not in cache:
                D = _Dense(nt, pt[0], pt[1], pt[4], dev)
                fac = _factored(D)
                cache[key] = (D, fac, _first_order(D, fac)[0])
            D, fac, lam = cache[key]
            out.append(_second_order(D, fac, lam, torch.as_tensor(np.ascontiguousarray(w), device=dev)))
        return out
    vm, va, x, p, pd, qd = d["points"][0]
    if kind == "resolve":
        return [_newton(net, vm, va, p, pd * s, qd * s, dev)[2] for s in d["scales"]]
    if kind == "newton_cg":
        out, v = [], torch.as_tensor(d["w"][:, :1].copy(), device=dev)
        for q in (p, d["p1"]):
            vq, aq, _ = _newton(net, vm, va, q, pd, qd, dev)
            D = _Dense(net, vq, aq, pd, dev)
            fac = _factored(D)
            lam, grad = _first_order(D, fac)
            out += [torch.tensor(D.F, dtype=torch.float64), grad, _second_order(D, fac, lam, v)[:, 0]]
        return out
    if kind == "track":
        s = d["scales"][0]
        pd, qd = pd * s, qd * s
        vm, va, x = _newton(net, vm, va, p, pd, qd, dev)
    D = _Dense(net, vm, va, pd, dev)
    fac = _factored(D)
    if kind == "solve":
        return _solve(fac[3], fac[0], torch.as_tensor(np.ascontiguousarray(d["r"]), device=dev), case["trans"])
    lam, grad = _first_order(D, fac)
    if kind == "adjoint":
        return lam, grad, D.F
    if kind == "hessvec":
        return _second_order(D, fac, lam, torch.as_tensor(np.ascontiguousarray(d["w"]), device=dev))
    H = _second_order(D, fac, lam, torch.eye(net.n_p, dtype=torch.float64, device=dev))
    if kind == "hessian":
        return H, grad, D.F
    L = torch.linalg.cholesky((H + H.t()) / 2)
    step = torch.cholesky_solve(-grad[:, None], L)[:, 0]
    return x, lam, grad, D.F, step, torch.as_tensor(p, device=dev) + step, torch.tril(L) + torch.triu(H, 1), None
