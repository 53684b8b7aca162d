"""Unit form of the tree solve (csrc/units.cu) at the shapes where it can go
wrong: one unit and one vertex more, units of the smallest size and ragged
last ones, three levels, hubs whose contribution lists and export lists are
long, deep paths and trees that branch everywhere, against the oracle's
solve.

Tolerances: FP64 as the other tree-solve tests (1e-10 of max |x|); FP32 1e-4
of max |x|: a value passes at most 3 levels x 2 x about 14 rounds of
additions of terms of its own size, 84 x 2^-24 = 5e-6, and 20 times that is
left for cancellation in right-hand sides of zero mean.
"""
import numpy as np
import pytest

import oracle
from synth import graphs, rng
from tests.gpu_util import dev, gpu_graph, host

pytestmark = pytest.mark.gpu


def _tree(kind, n, seed):
    """Parent of every vertex (0: root), before the ids are shuffled."""
    i = np.arange(n, dtype=np.int64)
    u = rng.uniform(seed, 1, n)
    if kind == "path":
        return np.maximum(i - 1, 0)
    if kind == "star":
        return np.zeros(n, dtype=np.int64)
    if kind == "heap":
        return np.maximum((i - 1) // 2, 0)
    if kind == "random":
        return (u * i).astype(np.int64)
    if kind == "caterpillar":                       # a spine with three legs a vertex
        return np.where(i % 4 == 0, np.maximum(i - 4, 0), i - i % 4)
    if kind == "brooms":                            # 40 hubs along a path, the rest leaves
        return np.where(i < 40, np.maximum(i - 1, 0), i % 40)
    raise ValueError(kind)


def _graph(kind, n, seed):
    par = _tree(kind, n, seed)
    perm = np.argsort(rng.uniform(seed, 2, n), kind="stable")
    a, b = perm[np.arange(1, n)], perm[par[1:]]
    w = 10.0 ** (2.0 * rng.uniform(seed, 3, n - 1) - 1.0)
    rp, col, val = graphs.csr_from_edges(n, np.minimum(a, b), np.maximum(a, b), w,
                                         1e-3 * rng.uniform(seed, 4, n))
    return graphs.Graph(f"{kind}{n}", n, rp, col, val)


CASES = [("path", 2), ("path", 3), ("path", 3584), ("path", 3585), ("path", 20011),
         ("star", 700), ("star", 9001), ("star", 60013), ("heap", 4097), ("heap", 65535),
         ("random", 3585), ("random", 7681), ("random", 272300), ("random", 300007), ("caterpillar", 12001),
         ("brooms", 50021)]


@pytest.mark.parametrize("kind,n", CASES)
@pytest.mark.parametrize("r,prec", [(1, "fp64"), (2, "fp32"), (4, "fp64"), (8, "fp64"), (16, "fp32"), (24, "fp32"), (24, "fp64")])
def test_unit_solve_matches_oracle(gpu, kind, n, r, prec):
    import torch
    g = _graph(kind, n, 7)
    rho = n // 3
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og, rho)
    P, dt, tol = ((gpu.GRASS_FP64, torch.float64, 1e-10) if prec == "fp64"
                  else (gpu.GRASS_FP32, torch.float32, 1e-4))
    B = rng.gaussian_block(5, 6, n, r).astype(np.float32).astype(np.float64)
    with gpu_graph(g, rho) as (ctx, tree, _):
        Bd = dev(B, dt)
        # a right-hand side and a solution that are not 16-byte aligned
        odd = torch.empty(n * r + 1, dtype=dt, device="cuda")[1:].view(n, r)
        odd.copy_(Bd)
        for with_D in (0, 1):
            # the grounded solve does not depend on B[rho]; a zero sum lets the
            # oracle refine its answer
            B0 = B.copy()
            B0[rho] -= B.sum(axis=0)
            ref = oracle.tree_solve(og, ot, B, og.D) if with_D else oracle.tree_solve(og, ot, B0)
            X = torch.full_like(Bd, float("nan"))
            gpu.grass_tree_solve(ctx, tree, with_D, r, P, Bd, X)
            x = host(X).astype(np.float64)
            assert np.abs(x - ref).max() <= tol * np.abs(ref).max(), with_D
            if not with_D:
                assert np.all(x[rho] == 0.0)
            # the same bits in place, unaligned, and with another launch shape
            gpu.grass_ctx_set_param(ctx, "tree_threads", 160)
            gpu.grass_tree_solve(ctx, tree, with_D, r, P, odd, odd)
            gpu.grass_ctx_set_param(ctx, "tree_threads", 1024)
            scan = r == 1 and not with_D      # the scan form's block sums follow the launch shape
            assert scan or torch.equal(odd, X), with_D
            odd.copy_(Bd)


@pytest.mark.parametrize("n", [3, 3585, 20011])
def test_round_sizes_on_demand(gpu, n):
    """The elimination rounds' sizes of a tree that solves in units: those of
    the same tree as a batch of one, and after the query the tree solves as
    before it and holds no more device memory."""
    import torch
    g = _graph("random", n, 8)
    B = dev(rng.gaussian_block(5, 7, n, 4))
    X, Y = torch.empty_like(B), torch.empty_like(B)
    with gpu_graph(g, 0) as (ctx, tree, csr):
        forest = gpu.grass_build_forest(ctx, *csr, [0, n])
        try:
            sizes = gpu.grass_tree_schedule_info(forest)
            assert gpu.grass_tree_info(forest) == (n, n - 1, len(sizes[0])) and sum(sizes[0]) == n - 1
        finally:
            gpu.grass_tree_destroy(forest)
        assert gpu.grass_tree_info(tree, rounds=False)[:2] == (n, n - 1)
        gpu.grass_tree_solve(ctx, tree, 1, 4, gpu.GRASS_FP64, B, X)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        assert gpu.grass_tree_schedule_info(tree) == sizes
        assert gpu.grass_tree_info(tree) == (n, n - 1, len(sizes[0]))
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
        gpu.grass_tree_solve(ctx, tree, 1, 4, gpu.GRASS_FP64, B, Y)
        assert torch.equal(X, Y)


def test_autotune_leaves_the_tail_of_a_tree_without_one(gpu):
    """A single tree's solve has no tail to tune: the forests' setting stays."""
    g = _graph("random", 7681, 8)
    with gpu_graph(g, 0) as (ctx, tree, _):
        for tail in (777, 20000):
            gpu.grass_ctx_set_param(ctx, "tree_tail_items", tail)
            for r in (1, 8):
                best, ms = gpu.grass_autotune(ctx, tree, r, gpu.GRASS_FP32)
                assert best[2] == tail and best[0] in (256, 512, 1024) and ms > 0


@pytest.mark.parametrize("kind,n", [("random", 20011), ("star", 9001), ("random", 280001)])
@pytest.mark.parametrize("r,prec", [(16, "fp64"), (32, "fp64"), (32, "fp32")])
def test_unit_solve_in_column_groups(gpu, kind, n, r, prec):
    """More than one column group a unit, with units in number below and (on 4
    SMs, or from 272,384 vertices on) above the grid's thread groups."""
    import torch
    g = _graph(kind, n, 9)
    rho = n // 3
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og, rho)
    P, dt, tol = ((gpu.GRASS_FP64, torch.float64, 1e-10) if prec == "fp64"
                  else (gpu.GRASS_FP32, torch.float32, 1e-4))
    B = rng.gaussian_block(5, 8, n, r).astype(np.float32).astype(np.float64)
    ref = oracle.tree_solve(og, ot, B, og.D)
    with gpu_graph(g, rho) as (ctx, tree, _):
        Bd = dev(B, dt)
        X, Y = torch.full_like(Bd, float("nan")), torch.full_like(Bd, float("nan"))
        gpu.grass_tree_solve(ctx, tree, 1, r, P, Bd, X)
        assert np.abs(host(X).astype(np.float64) - ref).max() <= tol * np.abs(ref).max()
        gpu.grass_ctx_set_param(ctx, "grid_sms", 4)
        gpu.grass_tree_solve(ctx, tree, 1, r, P, Bd, Y)
        assert torch.equal(X, Y)
