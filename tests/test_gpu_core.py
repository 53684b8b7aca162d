"""CG on the sparsifier's core (csrc/core.cu) against the oracle's CG over
all vertices: the same iterates, so the same embedding both when the solves
converge and when every one ends at its iteration cap, on trees whose core is
a single unit and several, with hubs, doubled edges' ends and every column
count; and the sides of the rule that chooses it.

Tolerances: FP64 1e-10 of the largest heat, as the other embedding tests (the
capped iterates are those of exact arithmetic up to rounding on both sides);
FP32 1e-3 as there.
"""
import numpy as np
import pytest

import oracle
from synth import graphs, rng
from tests.gpu_util import dev, gpu_graph, host
from tests.test_gpu_parity import _densify_parity

pytestmark = pytest.mark.gpu


def _graph(kind):
    if kind == "grid3d":
        return graphs.grid3d_loguniform(22, 21, 20, seed=3)
    if kind == "power":
        return graphs.power_grid(70, seed=4)
    if kind == "mesh":
        return graphs.grid2d_uniform(181, 160, seed=5, lo=0.1, hi=10.0)
    return graphs.chung_lu(6000, seed=6)


@pytest.mark.parametrize("kind,every", [("grid3d", 97), ("power", 61), ("mesh", 211), ("mesh", 4001),
                                        ("powerlaw", 401)])
@pytest.mark.parametrize("maxit,tol", [(3000, 1e-13), (4, 1e-13)])
@pytest.mark.parametrize("r", [2, 8, 16, 24])
def test_core_embedding_matches_oracle(gpu, kind, every, maxit, tol, r):
    import torch
    g = _graph(kind)
    og = oracle.from_graph(g)
    rho = g.n // 2
    ot = oracle.build_tree(og, rho)
    off = np.flatnonzero(ot.in_tree == 0)
    add = off[::every]
    in_s = ot.in_tree.copy()
    in_s[add] = 1
    h0 = rng.gaussian_block(11, 3, g.n, r)
    H = oracle.embed(og, ot, in_s, h0, 1, tol, maxit)
    heat_ref, _ = oracle.heat(og, in_s, H)
    with gpu_graph(g, rho) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add.astype(np.int64)))
            for P, dt, bound in ((gpu.GRASS_FP64, torch.float64, 1e-10), (gpu.GRASS_FP32, torch.float32, 1e-3)):
                if P == gpu.GRASS_FP32 and maxit > 100:
                    t2, m2 = 1e-6, 200
                else:
                    t2, m2 = tol, maxit
                heat = torch.empty(heat_ref.shape[0], dtype=dt, device="cuda")
                hm = gpu.grass_embed(ctx, S, dev(h0), r, 1, P, t2, m2, None, heat)
                x = host(heat).astype(np.float64)
                assert np.abs(x - heat_ref).max() <= bound * heat_ref.max(), P
                assert hm == pytest.approx(heat_ref.max(), rel=bound)
        finally:
            gpu.grass_sparsifier_destroy(S)


@pytest.mark.parametrize("added", [1, 126, 128, 129, 200])
def test_rule_sides_agree(gpu, added):
    """45 x 46 = 2070 vertices: up to 129 added edges take the core, more the
    CG over all vertices; adding edges to S rebuilds it."""
    import torch
    g = graphs.grid2d_uniform(45, 46, seed=9)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    off = np.flatnonzero(ot.in_tree == 0)
    h0 = rng.gaussian_block(12, 3, g.n, 4)
    with gpu_graph(g) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            for part in (off[:max(1, added // 2)], off[:added]):
                gpu.grass_sparsifier_add(ctx, S, dev(part.astype(np.int64)))
                in_s = ot.in_tree.copy()
                in_s[part] = 1
                H = oracle.embed(og, ot, in_s, h0, 2, 1e-13, 2000)
                heat_ref, _ = oracle.heat(og, in_s, H)
                heat = torch.empty(heat_ref.shape[0], dtype=torch.float64, device="cuda")
                gpu.grass_embed(ctx, S, dev(h0), 4, 2, gpu.GRASS_FP64, 1e-13, 2000, None, heat)
                assert np.abs(host(heat) - heat_ref).max() <= 1e-10 * heat_ref.max()
        finally:
            gpu.grass_sparsifier_destroy(S)


def _core_at_least(g, ot, in_s):
    """A lower bound of the core's size: the vertices of the tree that rake and
    compress leave when the ends of the added edges must stay (the ends and the
    branchings of the paths between them; unit borders come on top)."""
    added = np.flatnonzero((in_s != 0) & (ot.in_tree == 0))
    og = oracle.from_graph(g)
    pin = np.zeros(g.n, dtype=bool)
    pin[og.eu[added]] = pin[og.ev[added]] = True
    # paths that reach a vertex from below: 2 and more make it a branching
    below = np.zeros(g.n, dtype=np.int64)
    core = pin.copy()
    for v in ot.order[::-1]:
        core[v] |= below[v] >= 2
        p = ot.parent[v]
        if p >= 0 and (core[v] or below[v]):
            below[p] += 1
    return int(core.sum())


def test_densify_core_larger_than_the_edge_list(gpu):
    """Two FP64 rounds of 32 columns with a 5 % cap on a new context: round 2's
    inner solves run on the core, whose block is larger than the list of
    accepted edge ids that the rounds keep."""
    g = graphs.grid2d_uniform(90, 80, seed=21)
    cap, r = g.n // 20, 32
    d, res = _densify_parity(gpu, g, 5.0, r, 2, 2, cap)
    assert d["rounds"] == 2 and d["added_round"] == res.added
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    in_s = ot.in_tree.copy()      # S in round 2
    in_s[oracle.filter_edges(res.trace[0]["heat"], res.trace[0]["off"], res.theta[0], cap)] = 1
    assert g.n >= 2048 and 16 * cap <= g.n and _core_at_least(g, ot, in_s) * r * 8 > 8 * (og.m + 1) + 256


def _on_core(gpu, ctx, S, n, h0, r, prec, maxit=160, t=1):
    """Whether S's inner solves of `maxit` iterations run on its core, from the
    algorithmic bytes of the kernel-family timing: an iteration over all
    vertices moves at least 14 n-row blocks (the CG's vectors 12, the product and
    the tree solve 2 each, 2 less in the first), one on the core about 17 of its
    own rows, a quarter of n at most, and its indices."""
    gpu.grass_kernel_timing_enable(ctx, gpu.GRASS_KF_CG)
    gpu.grass_embed(ctx, S, h0, r, t, prec, 0.0, maxit)
    _, launches, by = gpu.grass_kernel_timing_read(ctx)
    gpu.grass_kernel_timing_enable(ctx, gpu.GRASS_KF_NONE)
    blocks = by / (n * r * (8 if prec == gpu.GRASS_FP64 else 4)) / (maxit * t)
    assert launches == t and (blocks >= 14 or blocks <= 10)
    return blocks <= 10


def _fill_device(torch, leave):
    """Tensors that take the free device memory up to about `leave` bytes."""
    held, size = [], torch.cuda.mem_get_info()[0] - leave
    while size >= 1 << 21:
        try:
            held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            size //= 2
            continue
        size = min(size, torch.cuda.mem_get_info()[0] - leave)
    return held


@pytest.mark.parametrize("leave_mb", [3, 6, 10])
def test_core_without_room_serves_over_all_vertices(gpu, leave_mb):
    """Device memory that ends somewhere in the core's construction (at least 13
    MB here): the call is served by the CG over all vertices, the repeated one
    too, and S has its core again once it has changed and there is room."""
    import torch
    g = graphs.grid2d_uniform(300, 301, seed=23)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    off = np.flatnonzero(ot.in_tree == 0)
    h0 = rng.gaussian_block(13, 3, g.n, 2)
    h0d, FP64 = dev(h0), gpu.GRASS_FP64
    few, many = dev(off[::97].astype(np.int64)), dev(off[::5].astype(np.int64))
    in_s = ot.in_tree.copy()
    in_s[off[::97]] = 1
    ref, _ = oracle.heat(og, in_s, oracle.embed(og, ot, in_s, h0, 1, 1e-13, 3000))
    heat = torch.empty(ref.shape[0], dtype=torch.float64, device="cuda")
    with gpu_graph(g) as (ctx, tree, _):
        made = []

        def sparsifier(ids):
            S = gpu.grass_sparsifier_create(ctx, tree)
            made.append(S)
            gpu.grass_sparsifier_add(ctx, S, ids)
            return S

        def right(S):
            heat.fill_(float("nan"))
            gpu.grass_embed(ctx, S, h0d, 2, 1, FP64, 1e-13, 3000, None, heat)
            assert np.abs(host(heat) - ref).max() <= 1e-10 * ref.max()

        try:
            # both forms' kernels, scratch and timing buffers first
            assert _on_core(gpu, ctx, sparsifier(few), g.n, h0d, 2, FP64)
            assert not _on_core(gpu, ctx, sparsifier(many), g.n, h0d, 2, FP64)
            S = sparsifier(few)
            host(heat.fill_(0.0))
            torch.cuda.synchronize()
            held = _fill_device(torch, leave_mb << 20)
            try:
                right(S)
                right(S)
                small = not _on_core(gpu, ctx, S, g.n, h0d, 2, FP64)
            finally:
                del held
                torch.cuda.empty_cache()
            assert small
            right(S)
            gpu.grass_sparsifier_add(ctx, S, dev(off[1:2].astype(np.int64)))
            assert _on_core(gpu, ctx, S, g.n, h0d, 2, FP64)
        finally:
            for S in made:
                gpu.grass_sparsifier_destroy(S)


@pytest.mark.parametrize("side,r,prec,maxit,t,core", [
    (60, 2, "fp64", 8, 1, False), (60, 2, "fp64", 63, 1, False), (60, 2, "fp64", 64, 1, True),
    (60, 2, "fp64", 32, 2, True), (300, 2, "fp32", 159, 1, False), (300, 2, "fp32", 160, 1, True),
    (300, 32, "fp64", 5, 1, False), (300, 32, "fp64", 6, 1, True), (300, 32, "fp64", 3, 2, True),
    (300, 32, "fp32", 22, 1, False), (300, 32, "fp32", 23, 1, True)])
def test_core_waits_for_iterations_that_pay_its_build(gpu, side, r, prec, maxit, t, core):
    """The rule's sides in the iterations a call allows: 64 in FP64 and 160 in
    FP32, or 128 and 256 MB over the block's bytes (23 and 11.5 MB here)."""
    P = gpu.GRASS_FP64 if prec == "fp64" else gpu.GRASS_FP32
    g = graphs.grid2d_uniform(side, side, seed=9)
    ot = oracle.build_tree(oracle.from_graph(g))
    add = np.flatnonzero(ot.in_tree == 0)[::97].astype(np.int64)
    with gpu_graph(g) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add))
            h0 = dev(rng.gaussian_block(12, 3, g.n, r))
            assert _on_core(gpu, ctx, S, g.n, h0, r, P, maxit, t) == core
        finally:
            gpu.grass_sparsifier_destroy(S)


@pytest.mark.parametrize("r,prec", [(8, "fp64"), (16, "fp64"), (24, "fp64"), (32, "fp64"),
                                    (16, "fp32"), (24, "fp32"), (32, "fp32")])
@pytest.mark.parametrize("sms", [0, 4])
def test_core_columns_in_groups(gpu, r, prec, sms):
    """Every count of column groups a unit is worked on in, spread over the grid
    (sms = 0: more thread groups than units) and one after the other in the
    group that has staged the unit's lists (4 SMs: fewer)."""
    import torch
    g = graphs.grid3d_loguniform(22, 21, 20, seed=3)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    add = np.flatnonzero(ot.in_tree == 0)[::97]
    in_s = ot.in_tree.copy()
    in_s[add] = 1
    h0 = rng.gaussian_block(11, 4, g.n, r)
    ref, _ = oracle.heat(og, in_s, oracle.embed(og, ot, in_s, h0, 1, 1e-13, 3000))
    P, dt, bound, tol, maxit = ((gpu.GRASS_FP64, torch.float64, 1e-10, 1e-13, 3000) if prec == "fp64"
                                else (gpu.GRASS_FP32, torch.float32, 1e-3, 1e-6, 200))
    with gpu_graph(g) as (ctx, tree, _):
        gpu.grass_ctx_set_param(ctx, "grid_sms", sms)
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add.astype(np.int64)))
            heat = torch.empty(ref.shape[0], dtype=dt, device="cuda")
            gpu.grass_embed(ctx, S, dev(h0), r, 1, P, tol, maxit, None, heat)
            assert np.abs(host(heat).astype(np.float64) - ref).max() <= bound * ref.max()
            assert _on_core(gpu, ctx, S, g.n, dev(h0), r, P)
        finally:
            gpu.grass_sparsifier_destroy(S)


@pytest.mark.parametrize("added,core", [(126, True), (128, True), (129, True), (130, False), (200, False)])
def test_core_rule_in_added_edges(gpu, added, core):
    """2070 vertices: 129 added edges are the last that take the core."""
    g = graphs.grid2d_uniform(45, 46, seed=9)
    ot = oracle.build_tree(oracle.from_graph(g))
    add = np.flatnonzero(ot.in_tree == 0)[:added].astype(np.int64)
    with gpu_graph(g) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add))
            assert _on_core(gpu, ctx, S, g.n, dev(rng.gaussian_block(12, 3, g.n, 4)), 4, gpu.GRASS_FP64) == core
        finally:
            gpu.grass_sparsifier_destroy(S)


def test_core_capped_solve_of_a_large_graph(gpu):
    """Solves that end at their cap on the core (8 iterations): the iterate is
    the oracle's.  Tolerance: a start block moved by 1e-15 moves the oracle's own
    heats by 6e-12 of the largest here; rounding moves the vectors of 8
    iterations by up to some 1e-13, a hundred times that, and 1e-8 leaves a
    factor of 16 (one iteration more changes 0.8)."""
    import torch
    g = graphs.grid2d_uniform(725, 724, seed=21)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    add = np.flatnonzero(ot.in_tree == 0)[::17]
    in_s = ot.in_tree.copy()
    in_s[add] = 1
    h0 = rng.gaussian_block(11, 5, g.n, 8)
    ref, _ = oracle.heat(og, in_s, oracle.embed(og, ot, in_s, h0, 1, 1e-13, 8))
    with gpu_graph(g) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add.astype(np.int64)))
            heat = torch.empty(ref.shape[0], dtype=torch.float64, device="cuda")
            gpu.grass_embed(ctx, S, dev(h0), 8, 1, gpu.GRASS_FP64, 1e-13, 8, None, heat)
            assert np.abs(host(heat) - ref).max() <= 1e-8 * ref.max()
            assert _on_core(gpu, ctx, S, g.n, dev(h0), 8, gpu.GRASS_FP64, 8)
        finally:
            gpu.grass_sparsifier_destroy(S)


def test_core_above_a_quarter_is_not_used(gpu):
    """A binary tree of 262 leaves whose 522 branches are chains of three
    vertices, the leaves joined in pairs by 131 added edges: ends and branchings
    are a quarter of the 2096 vertices less one, the cuts between units lie on
    chains and add to them."""
    import torch
    n, k = 2096, 131
    heap = np.arange(1, 523)
    first = 523 + 3 * (heap - 1)                       # the chain above heap vertex h
    par = np.zeros(n, dtype=np.int64)
    par[heap], par[first], par[first + 1], par[first + 2] = first + 2, (heap - 1) // 2, first, first + 1
    par[2089:] = np.arange(2088, 2095)                 # the rest on one more chain
    i, leaves = np.arange(1, n), np.arange(261, 523)
    u, v = np.concatenate([par[1:], leaves[:k], [0]]), np.concatenate([i, leaves[k:], [n - 1]])
    w = np.concatenate([10.0 + rng.uniform(3, 1, n - 1), 1.0 + rng.uniform(3, 2, k + 1)])
    g = graphs.Graph("leaves", n, *graphs.csr_from_edges(n, u, v, w, 1e-3))
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    in_s = ot.in_tree.copy()
    add = np.flatnonzero((ot.in_tree == 0) & (og.eu >= 261))
    in_s[add] = 1                                      # one edge stays outside S
    h0 = rng.gaussian_block(12, 3, n, 4)
    ref, off = oracle.heat(og, in_s, oracle.embed(og, ot, in_s, h0, 1, 1e-13, 2000))
    assert add.size == k and off.size == 1 and 4 * (_core_at_least(g, ot, in_s) + 1) == n
    with gpu_graph(g) as (ctx, tree, _):
        S = gpu.grass_sparsifier_create(ctx, tree)
        try:
            gpu.grass_sparsifier_add(ctx, S, dev(add.astype(np.int64)))
            heat = torch.empty(1, dtype=torch.float64, device="cuda")
            gpu.grass_embed(ctx, S, dev(h0), 4, 1, gpu.GRASS_FP64, 1e-13, 2000, None, heat)
            assert np.abs(host(heat) - ref).max() <= 1e-10 * ref.max()
            assert not _on_core(gpu, ctx, S, n, dev(h0), 4, gpu.GRASS_FP64)
        finally:
            gpu.grass_sparsifier_destroy(S)
