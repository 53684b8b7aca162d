"""Performance cases of the sparsify-and-solve library, called as a program calls it.

A case names a graph family, its size and the call that is made on it; every
family is one that the tests and the benchmark use:

  grid2d   5-point grid, w in [1, 10), D = 1e-3 (meshes; the latency config)
  grid3d   7-point grid, w = 10^U(-2, 2), D = 1e-3 (FEM / thermal matrices)
  power    5-point grid, w in [0.1, 10], 1 % long-range vias of weight 100,
           pad loads in [1e-4, 1e-2] (power grids)
  mesh     5-point grid of unit weights, D = 0 (partitioning, low-stretch tree)
  powerlaw unit-weight graph with Chung-Lu degrees (networks, hub vertices)
  batch    a union of grids and of rings with chords (many systems at once)

and every call is an entry point of include/grass.h.  Weights and loads are
multiples of 2^-20, so that row sums are exact in any order.  Systems are
solved to a residual far below the one of everyday use, so that the answer is
a property of the system and not of the path the iteration took.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1911_04382_gb300 as G

DEV = "cuda"
Q = float(1 << 20)   # weights are multiples of 1 / Q


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _grid_edges(dims):
    """Edges of a grid (vertex id = x + dims[0] (y + dims[1] z))."""
    n = math.prod(dims)
    ids = torch.arange(n, device=DEV)
    us, vs, stride, rem = [], [], 1, ids
    for d in dims:
        u = ids[rem % d < d - 1]
        us.append(u)
        vs.append(u + stride)
        stride *= d
        rem = rem // d
    return n, torch.cat(us), torch.cat(vs)


def _distinct(n, a, b):
    """The distinct pairs a != b as (smaller, larger), by increasing pair."""
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    key = torch.unique(lo[lo != hi] * n + hi[lo != hi])
    return key // n, key % n


def _quant(w):
    return torch.clamp(torch.round(w * Q), min=1.0) / Q


def _ring_chords(n, gen):
    i = torch.arange(n, device=DEV)
    k = max(1, n // 4)
    a = torch.randint(0, n, (k,), generator=gen, device=DEV)
    b = torch.randint(0, n, (k,), generator=gen, device=DEV)
    return _distinct(n, torch.cat([i, a]), torch.cat([(i + 1) % n, b]))


def _sizes(case):
    """Sides / sizes of the graphs of a batch: spread over a factor of 16."""
    k, top = case["count"], case["size"]
    return [max(64, int(top * 16.0 ** (-(j // 2) / max(1, (k - 1) // 2)))) for j in range(k)]


def _edges(case, seed):
    """(n, u, v, w, D, graph offsets) of a case, edges by increasing (u, v)."""
    gen, kind = _gen(seed), case["graph"]
    rand = lambda k: torch.rand(k, generator=gen, device=DEV, dtype=torch.float64)  # noqa: E731
    off, D = None, 1e-3
    if kind in ("grid2d", "mesh"):
        n, u, v = _grid_edges((case["nx"], case["ny"]))
    elif kind == "grid3d":
        n, u, v = _grid_edges((case["nx"], case["ny"], case["nz"]))
    elif kind == "power":
        n, u, v = _grid_edges((case["nx"], case["ny"]))
        k = max(1, n // 100)
        a = torch.randint(0, n, (k,), generator=gen, device=DEV)
        b = torch.randint(0, n, (k,), generator=gen, device=DEV)
        a, b = _distinct(n, a, b)
        dx, dy = (a % case["nx"] - b % case["nx"]).abs(), (a // case["nx"] - b // case["nx"]).abs()
        far = dx + dy > 1   # not neighbours on the grid
        via = torch.cat([torch.zeros_like(u), torch.ones_like(a[far])]).bool()
        u, v = torch.cat([u, a[far]]), torch.cat([v, b[far]])
    elif kind == "powerlaw":
        # a random attachment tree (so that the graph is connected) and
        # Chung-Lu endpoints of exponent 2.1, mean degree 10
        n = case["n"]
        wt = (torch.arange(n, device=DEV, dtype=torch.float64) + 1.0) ** (-1.0 / 1.1)
        wt = torch.clamp(wt * (10.0 * n / wt.sum()), max=math.sqrt(10.0 * n))
        cdf = torch.from_numpy(np.cumsum(wt.cpu().numpy())).to(DEV)
        ends = torch.searchsorted(cdf / cdf[-1], rand(8 * n), right=True).clamp(max=n - 1)
        i = torch.arange(1, n, device=DEV)
        parent = (rand(n - 1) * i).long().minimum(i - 1)
        u, v = _distinct(n, torch.cat([ends[0::2], i]), torch.cat([ends[1::2], parent]))
    else:   # batch: even graphs are grids, odd ones rings with chords
        n, us, vs, off = 0, [], [], [0]
        for j, s in enumerate(_sizes(case)):
            if j % 2 == 0:
                side = max(8, int(math.sqrt(s)))
                k, a, b = _grid_edges((side, side + 1))
            else:
                k = s
                a, b = _ring_chords(k, gen)
            us.append(a + n)
            vs.append(b + n)
            n += k
            off.append(n)
        u, v = torch.cat(us), torch.cat(vs)
    order = torch.argsort(u * n + v)
    u, v, m = u[order], v[order], u.numel()
    if kind in ("mesh", "powerlaw"):
        w, D = torch.ones(m, device=DEV, dtype=torch.float64), 0.0
    elif kind == "grid3d":
        w = 10.0 ** (4.0 * rand(m) - 2.0)
    elif kind == "power":
        w = torch.where(via[order], 100.0, 0.1 + 9.9 * rand(m))
        D = 1e-4 + 9.9e-3 * rand(n)
    else:
        w = 1.0 + 9.0 * rand(m)
    D = torch.zeros(n, device=DEV, dtype=torch.float64) + D
    return n, u, v, _quant(w), torch.round(D * Q) / Q, off


def _csr(n, u, v, w, D):
    """Full symmetric CSR of L_G + diag(D), rows sorted by column."""
    i = torch.arange(n, device=DEV)
    deg = torch.zeros(n, device=DEV, dtype=torch.float64)
    deg.index_add_(0, u, w).index_add_(0, v, w)
    rows = torch.cat([u, v, i])
    cols = torch.cat([v, u, i])
    vals = torch.cat([-w, -w, deg + D])
    order = torch.argsort(rows * n + cols)
    ptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return ptr, cols[order].to(torch.int32), vals[order]


def _normal(case, seed, salt, *shape):
    return torch.randn(*shape, generator=_gen(seed * 16 + salt), device=DEV, dtype=torch.float64)


def _extra(case, seed, m):
    """Edge ids a sparsifier gets on top of its tree (2 % of the vertices)."""
    k = max(4, m // 60)
    return torch.unique(torch.randint(0, m, (k,), generator=_gen(seed * 16 + 7), device=DEV))


def _heat_room(case):
    """Room for the heats of any graph of this family and size."""
    if case["graph"] == "powerlaw":
        return 5 * case["n"]
    return (3 if case["graph"] == "grid3d" else 2) * math.prod(
        case[k] for k in ("nx", "ny", "nz") if k in case)


# ---------------------------------------------------------------- cases

def listed():
    return [
        # the smallest whole call: one small FP64 system, all latency
        dict(name="solve_grid2d_64", call="solve", graph="grid2d", nx=64, ny=64, r=8, t=2,
             prec="fp64", rounds=1, cap=0.0, sigma2=100.0, precond="cg"),
        # one request of the serving form: a power grid, one round, 5 % cap
        dict(name="solve_power_301", call="solve", graph="power", nx=301, ny=301, r=8, t=2,
             prec="fp32", rounds=1, cap=0.05, sigma2=100.0, precond="tree"),
        # the largest whole call: three rounds and the multigrid PCG
        dict(name="solve_grid3d_100", call="solve", graph="grid3d", nx=100, ny=100, nz=100, r=16,
             t=2, prec="fp32", rounds=3, cap=0.02, sigma2=200.0, precond="amg"),
        # extraction, maximum spanning tree and its schedule alone
        dict(name="tree_grid3d_100", call="tree", graph="grid3d", nx=100, ny=100, nz=100),
        # the low-stretch tree of a unit mesh
        dict(name="lsst_mesh_500", call="lsst", graph="mesh", nx=500, ny=499),
        # the tree preconditioner of the PCG, one column, in FP64
        dict(name="tree_solve_power_1000_r1", call="tree_solve", graph="power", nx=1000, ny=1000,
             r=1, prec="fp64", with_D=True),
        # the grounded solve of the power iteration, 16 columns
        dict(name="tree_solve_grid3d_100_r16", call="tree_solve", graph="grid3d", nx=100, ny=100,
             nz=100, r=16, prec="fp32", with_D=False),
        # round 1 of densification: the embedding through the tree
        dict(name="embed_grid3d_100", call="embed", graph="grid3d", nx=100, ny=100, nz=100, r=16,
             t=2, prec="fp32", extra=False),
        # the same on a network with hubs, odd size, 24 columns, 3 steps
        dict(name="embed_powerlaw_200k", call="embed", graph="powerlaw", n=200003, r=24, t=3,
             prec="fp32", extra=False),
        # a later round in FP64: inner CG on the sparsifier, solved tightly
        dict(name="embed_extra_grid3d_50", call="embed", graph="grid3d", nx=50, ny=49, nz=51, r=8,
             t=2, prec="fp64", extra=True),
        # another right-hand side for a system whose sparsifier is kept
        dict(name="pcg_grid3d_100", call="pcg", graph="grid3d", nx=100, ny=100, nz=100, r=16, t=2,
             prec="fp32", rounds=3, cap=0.02, sigma2=200.0, precond="amg"),
        # 32 systems sparsified and solved in one batch
        dict(name="batch_32", call="batch", graph="batch", count=32, size=90000, r=8, t=2,
             prec="fp32", sigma2=100.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_case(rng, kind, lo, hi):
    n = _log(rng, lo, hi)
    if kind == "grid3d":
        a = max(4, int(n ** (1 / 3) * rng.uniform(0.7, 1.0)))
        b = max(4, int(math.sqrt(n / a)))
        return dict(graph=kind, nx=a, ny=b, nz=max(4, n // (a * b)))
    a = max(8, int(math.sqrt(n) * rng.uniform(0.6, 1.0)))
    return dict(graph=kind, nx=a, ny=max(8, n // a))


def draw(rng):
    call = rng.choice(["solve", "solve", "tree", "lsst", "tree_solve", "tree_solve", "embed",
                       "embed", "pcg", "batch"])
    if call in ("solve", "pcg"):
        c = _grid_case(rng, rng.choice(["grid2d", "grid3d", "power"]), 3e3, 7e5)
        c.update(r=rng.choice([4, 8, 16]), t=rng.choice([1, 2]), prec=rng.choice(["fp32", "fp64"]),
                 rounds=rng.choice([1, 2]), cap=rng.choice([0.02, 0.05]),
                 sigma2=rng.choice([100.0, 200.0]), precond=rng.choice(["tree", "amg"]))
    elif call == "tree":
        c = _grid_case(rng, rng.choice(["grid2d", "grid3d", "power"]), 1e3, 1e6)
    elif call == "lsst":
        c = _grid_case(rng, rng.choice(["mesh", "grid3d"]), 2e3, 2.5e5)
    elif call == "tree_solve":
        c = _grid_case(rng, rng.choice(["grid2d", "grid3d", "power"]), 2e3, 1e6)
        c.update(r=rng.choice([1, 2, 4, 8, 16, 24]), prec=rng.choice(["fp32", "fp64"]),
                 with_D=rng.choice([True, False]))
    elif call == "embed":
        extra = rng.choice([True, False])
        if extra:
            c = _grid_case(rng, rng.choice(["grid2d", "grid3d"]), 2e3, 1.2e5)
        elif rng.random() < 0.4:
            c = dict(graph="powerlaw", n=_log(rng, 5e3, 4e5))
        else:
            c = _grid_case(rng, rng.choice(["grid2d", "grid3d", "power"]), 2e3, 1e6)
        c.update(r=rng.choice([8, 16, 24]), t=rng.choice([1, 2]), extra=extra,
                 prec="fp64" if extra else rng.choice(["fp32", "fp64"]))
    else:
        c = dict(graph="batch", count=rng.randint(8, 40), size=_log(rng, 4e3, 9e4), r=8, t=2,
                 prec="fp32", sigma2=100.0)
    c["call"] = call
    return c


# ---------------------------------------------------------------- running

PREC = {"fp64": G.GRASS_FP64, "fp32": G.GRASS_FP32}
TOL = 1e-10          # PCG residual of every solve
INNER = (1e-13, 2000)  # inner CG of the tight FP64 embedding


class State:
    """A program's context, its handles and its device buffers."""

    def __init__(self, case):
        self.case = case
        self.ctx = G.grass_ctx_create()
        self.tree = self.S = None

    def __del__(self):
        for h, free in ((self.S, G.grass_sparsifier_destroy), (self.tree, G.grass_tree_destroy),
                        (self.ctx, G.grass_ctx_destroy)):
            if h:
                free(h)
        self.S = self.tree = self.ctx = None


def _params(case, n):
    cap = int(case["cap"] * n)
    fp64 = case["prec"] == "fp64"
    return G.make_params(case["sigma2"], case["r"], case["t"], case["rounds"], 8, cap,
                         PREC[case["prec"]], 1e-10 if fp64 else 1e-2, 1000 if fp64 else 30)


def prepare(case, seed):
    s = State(case)
    s.seed = seed
    n, u, v, w, D, off = _edges(case, seed)
    s.n, s.m, s.off = n, u.numel(), off
    s.csr = _csr(n, u, v, w, D)
    call, dt = case["call"], torch.float64 if case.get("prec") == "fp64" else torch.float32
    new = lambda *a, dtype=torch.float64: torch.empty(*a, device=DEV, dtype=dtype)  # noqa: E731
    if call in ("solve", "pcg", "batch"):
        k = case.get("rounds", 1)
        s.h0 = _normal(case, seed, 1, k * n, case["r"])
        s.v0 = _normal(case, seed, 2, k * n)
        s.b = _normal(case, seed, 3, n)
        s.x = new(n)
        G.grass_ctx_set_param(s.ctx, "pcg_precond", 1 if case.get("precond") == "amg" else 0)
    if call in ("tree", "lsst"):
        s.in_tree = new(s.m, dtype=torch.uint8)
    if call in ("tree_solve", "embed", "pcg"):
        s.tree = G.grass_build_tree(s.ctx, *s.csr, 0)
    if call == "tree_solve":
        s.b = _normal(case, seed, 3, n, case["r"]).to(dt)
        s.x = new(n, case["r"], dtype=dt)
    if call == "embed":
        s.S = G.grass_sparsifier_create(s.ctx, s.tree)
        if case["extra"]:
            G.grass_sparsifier_add(s.ctx, s.S, _extra(case, seed, s.m))
        s.h0 = _normal(case, seed, 1, n, case["r"])
        s.H = new(n, case["r"], dtype=dt)
        s.heat = new(_heat_room(case), dtype=dt).zero_()
    if call == "pcg":
        s.S, _ = G.grass_densify(s.ctx, s.tree, _params(case, n), s.h0, s.v0)
        del s.h0, s.v0
    return s


def _pcg(s, S):
    c = s.case
    st, info = G.grass_pcg_solve(s.ctx, S, s.b, s.x, TOL, 20000, PREC[c["prec"]], 1e-2, 1e-6,
                                 50 if c["precond"] == "cg" else 1)
    if st != G.GRASS_OK:
        raise RuntimeError("PCG did not reach its tolerance: %g" % info.rel_resid_fp64)
    return s.x


def run(s):
    c = s.case
    call = c["call"]
    if call == "tree_solve":
        G.grass_tree_solve(s.ctx, s.tree, int(c["with_D"]), c["r"], PREC[c["prec"]], s.b, s.x)
        return s.x
    if call == "embed":
        hmax = G.grass_embed(s.ctx, s.S, s.h0, c["r"], c["t"], PREC[c["prec"]], *INNER,
                             H_out=s.H, heat=s.heat)
        return {"H": s.H, "heat": s.heat, "heat_max": hmax}
    if call == "pcg":
        return _pcg(s, s.S)
    if call == "batch":
        tree = G.grass_build_forest(s.ctx, *s.csr, s.off)
    elif call == "lsst":
        tree, _ = G.grass_build_lsst(s.ctx, *s.csr, s.seed, 0)
    else:
        tree = G.grass_build_tree(s.ctx, *s.csr, 0)
    S = None
    try:
        if call in ("tree", "lsst"):
            G.grass_tree_edges(s.ctx, tree, s.in_tree)
            return s.in_tree
        if call == "batch":
            k = len(s.off) - 1
            P = G.make_params(c["sigma2"], c["r"], c["t"], 1, 8, 0, PREC[c["prec"]], 1e-2, 30)
            S, _, _ = G.grass_densify_batch(s.ctx, tree, P, s.h0, s.v0, k)
            st, info, _, _ = G.grass_pcg_solve_batch(s.ctx, S, s.b, s.x, TOL, 20000,
                                                     PREC[c["prec"]], 1, k)
            if st != G.GRASS_OK:
                raise RuntimeError("batch PCG missed its tolerance: %g" % info.rel_resid_fp64)
            return s.x
        S, _ = G.grass_densify(s.ctx, tree, _params(c, s.n), s.h0, s.v0)
        return _pcg(s, S)
    finally:
        if S:
            G.grass_sparsifier_destroy(S)
        G.grass_tree_destroy(tree)


def work(case):
    """Each input read once, each output written once; operations: those of
    one pass over the matrix entries and blocks (iterations not counted)."""
    k = case["graph"]
    if k == "powerlaw":
        n, m = case["n"], int(4.6 * case["n"])
    elif k == "batch":
        n = sum(_sizes(case))
        m = int(1.6 * n)
    elif k == "grid3d":
        n, m = case["nx"] * case["ny"] * case["nz"], 3 * case["nx"] * case["ny"] * case["nz"]
    else:
        n, m = case["nx"] * case["ny"], 2 * case["nx"] * case["ny"]
    csr = 8 * (n + 1) + 12 * (2 * m + n)
    call, r = case["call"], case.get("r", 1)
    es = 8 if case.get("prec") == "fp64" else 4
    if call in ("tree", "lsst"):
        return {"bytes": csr + m, "flops": 0}
    if call == "tree_solve":
        return {"bytes": 2 * n * r * es + n * (8 + 3 * es), "flops": 5 * n * r}
    if call == "embed":
        return {"bytes": 8 * n * r + n * r * es + 2 * m * (4 + es) + (m - n) * (8 + 2 * es),
                "flops": case["t"] * r * (6 * m + 5 * n) + 3 * r * (m - n)}
    if call == "pcg":
        return {"bytes": 2 * m * (4 + es) + 16 * n, "flops": 4 * m}
    return {"bytes": csr + case.get("rounds", 1) * n * (r + 1) * 8 + 16 * n,
            "flops": case["t"] * r * (6 * m + 5 * n)}


# ---------------------------------------------------------------- in 64 bits

class _TreeSolver:
    """L_T^{-1} (root 0 grounded) or (L_T + D)^{-1} of the maximum spanning
    tree, level by level from the leaves and back."""

    def __init__(self, n, u, v, w, D):
        m = u.numel()
        rank = torch.empty(m, device=DEV, dtype=torch.int64)
        rank[torch.argsort(w, descending=True, stable=True)] = torch.arange(m, device=DEV)
        comp = torch.arange(n, device=DEV)
        in_tree = torch.zeros(m, device=DEV, dtype=torch.bool)
        by_rank = torch.empty_like(rank)
        by_rank[rank] = torch.arange(m, device=DEV)
        while True:
            cu, cv = comp[u], comp[v]
            live = cu != cv
            if not bool(live.any()):
                break
            best = torch.full((n,), m, device=DEV, dtype=torch.int64)
            best.scatter_reduce_(0, cu[live], rank[live], "amin")
            best.scatter_reduce_(0, cv[live], rank[live], "amin")
            e = by_rank[best[best < m]]
            in_tree[e] = True
            while True:   # hook the larger label to the smaller, then shorten
                a, b = comp[u[e]], comp[v[e]]
                if bool((a == b).all()):
                    break
                comp.scatter_reduce_(0, torch.maximum(a, b), torch.minimum(a, b), "amin")
                while True:
                    nxt = comp[comp]
                    if bool((nxt == comp).all()):
                        break
                    comp = nxt
        self.in_tree = in_tree
        tu, tv, tw = u[in_tree], v[in_tree], w[in_tree]
        a, b, ww = torch.cat([tu, tv]), torch.cat([tv, tu]), torch.cat([tw, tw])
        order = torch.argsort(a)
        b, ww = b[order], ww[order]
        cnt = torch.bincount(a, minlength=n)
        ptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
        ptr[1:] = torch.cumsum(cnt, 0)
        par = torch.full((n,), -1, device=DEV, dtype=torch.int64)
        pw = torch.zeros(n, device=DEV, dtype=torch.float64)
        self.levels, front = [], torch.zeros(1, device=DEV, dtype=torch.int64)
        while True:
            c = cnt[front]
            at = torch.repeat_interleave(torch.arange(front.numel(), device=DEV), c)
            if at.numel() == 0:
                break
            first = torch.cumsum(c, 0) - c
            slot = ptr[front][at] + torch.arange(at.numel(), device=DEV) - first[at]
            p, q = front[at], b[slot]
            new = q != par[p]
            front = q[new]
            if front.numel() == 0:
                break
            par[front] = p[new]
            pw[front] = ww[slot[new]]
            self.levels.append(front)
        self.par, self.pw, dp = par, pw, D.clone()
        self.coef = torch.zeros(n, device=DEV, dtype=torch.float64)
        self.invd = torch.zeros(n, device=DEV, dtype=torch.float64)
        for f in reversed(self.levels):
            d = dp[f] + pw[f]
            self.coef[f], self.invd[f] = pw[f] / d, 1.0 / d
            dp.index_add_(0, par[f], dp[f] * self.coef[f])
        self.root = 1.0 / float(dp[0]) if float(dp[0]) > 0 else 0.0

    def __call__(self, B):
        x = B.clone()
        for f in reversed(self.levels):
            x.index_add_(0, self.par[f], x[f] * self.coef[f, None])
        x[0] *= self.root
        for f in self.levels:
            x[f] = x[f] * self.invd[f, None] + self.coef[f, None] * x[self.par[f]]
        return x


def _lap(n, u, v, w, D=None):
    """x -> L x (+ D x) for an n x r block, rows summed in a fixed order."""
    rows, cols = torch.cat([u, v]), torch.cat([v, u])
    vals = torch.cat([-w, -w])
    deg = torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, u, w).index_add_(0, v, w)
    diag = deg if D is None else deg + D
    order = torch.argsort(rows * n + cols)
    ptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    A = torch.sparse_csr_tensor(ptr, cols[order], vals[order], (n, n))
    return (lambda x: A @ x + diag[:, None] * x), diag


def _cg(mul, pre, B, tol, maxit):
    """CG on every column of B from zero, to a relative residual."""
    dot = lambda a, b: (a * b).sum(0)  # noqa: E731
    x, r = torch.zeros_like(B), B.clone()
    z = pre(r)
    p, rz, stop = z.clone(), dot(r, z), tol * tol * dot(B, B)
    for k in range(maxit):
        if k % 20 == 0 and bool((dot(r, r) <= stop).all()):
            break
        q = mul(p)
        pq = dot(p, q)
        a = torch.where(pq > 0, rz / pq, torch.zeros_like(pq))
        x += a * p
        r -= a * q
        z = pre(r)
        new = dot(r, z)
        p = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * p
        rz = new
    return x


def _refined(mul, pre, B, maxit):
    x = _cg(mul, pre, B, 1e-13, maxit)
    for _ in range(2):
        x += _cg(mul, pre, B - mul(x), 1e-6, maxit)
    return x


def exact(case, seed):
    call = case["call"]
    n, u, v, w, D, off = _edges(case, seed)
    if call in ("tree", "lsst"):
        return None   # whole numbers
    if call in ("solve", "pcg", "batch"):
        mul, diag = _lap(n, u, v, w, D)
        b = _normal(case, seed, 3, n)[:, None]
        return _refined(mul, lambda r: r / diag[:, None], b, 40000)[:, 0]
    if call == "tree_solve":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        T = _TreeSolver(n, u, v, w, D if case["with_D"] else torch.zeros_like(D))
        return T(_normal(case, seed, 3, n, case["r"]).to(dt).double())
    # the embedding: H <- L_S^{-1} L_G H, t times, and the off-S edges' heat
    T = _TreeSolver(n, u, v, w, torch.zeros_like(D))
    H = _normal(case, seed, 1, n, case["r"])
    in_s = T.in_tree.clone()
    if case["extra"]:
        in_s[_extra(case, seed, u.numel())] = True
        mulS, _ = _lap(n, u[in_s], v[in_s], w[in_s])

        def ground(x):
            return x - x[0:1]
        solve = lambda y: ground(_cg(mulS, T, y, 1e-15, 400))  # noqa: E731
    else:
        solve = T
    mulG, _ = _lap(n, u, v, w)
    for _ in range(case["t"]):
        H = solve(mulG(H))
        H = H * 2.0 ** (-math.floor(math.log2(float(H.abs().max()))))
    o = ~in_s
    hot = w[o] * (H[u[o]] - H[v[o]]).square().sum(1)
    heat = torch.zeros(_heat_room(case), device=DEV, dtype=torch.float64)
    heat[:hot.numel()] = hot
    return {"H": H, "heat": heat, "heat_max": float(hot.max())}
