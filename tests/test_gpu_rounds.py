"""The elimination rounds on a single tree (csrc/tree.cu, tree_solve.cuh), which
serve every tree above euler_max_n vertices: with that limit at 0 small graphs
take them too, in the stand-alone solves, the inner CG, the PCG's three forms
and the solve without allocation, each against the oracle, and against the unit
form that the same graph takes by default.

Tolerances: those of the same calls' other tests (FP64 solves 1e-10 of max |x|,
FP32 1e-4; heats 1e-10 of the largest; PCG its own residual).
"""
import contextlib

import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from synth import graphs, rng
from tests.gpu_util import dev, gpu_graph, host

pytestmark = pytest.mark.gpu


def _graph(kind):
    if kind == "grid2d":
        return graphs.grid2d_uniform(61, 60, seed=5)
    if kind == "grid3d":
        return graphs.grid3d_loguniform(22, 21, 20, seed=3)
    return graphs.chung_lu(6000, seed=6)


@contextlib.contextmanager
def _both(gpu, g, rho=0):
    """(ctx, tree in units, tree in rounds)"""
    with gpu_graph(g, rho) as (ctx, units, csr):
        gpu.grass_ctx_set_param(ctx, "euler_max_n", 0)
        rounds = gpu.grass_build_tree(ctx, *csr, rho)
        try:
            yield ctx, units, rounds
        finally:
            gpu.grass_tree_destroy(rounds)


@pytest.mark.parametrize("kind", ["grid2d", "grid3d", "powerlaw"])
@pytest.mark.parametrize("r,prec", [(1, "fp64"), (1, "fp32"), (8, "fp64"), (16, "fp32"), (32, "fp64")])
def test_solves(gpu, kind, r, prec):
    import torch
    g = _graph(kind)
    rho = g.n // 3
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og, rho)
    P, dt, tol = ((gpu.GRASS_FP64, torch.float64, 1e-10) if prec == "fp64"
                  else (gpu.GRASS_FP32, torch.float32, 1e-4))
    B = rng.gaussian_block(5, 6, g.n, r).astype(np.float32).astype(np.float64)
    # the grounded solve does not depend on B[rho]; a zero sum lets the oracle
    # refine its answer
    B0 = B.copy()
    B0[rho] -= B.sum(axis=0)
    Bd = dev(B, dt)
    with _both(gpu, g, rho) as (ctx, units, rounds):
        for with_D in (0, 1) if og.D.any() else (0,):
            ref = oracle.tree_solve(og, ot, B, og.D) if with_D else oracle.tree_solve(og, ot, B0)
            for solve in (gpu.grass_tree_solve, gpu.grass_tree_solve_noalloc):
                for tree in (rounds, units):
                    X = torch.full_like(Bd, float("nan"))
                    solve(ctx, tree, with_D, r, P, Bd, X)
                    assert np.abs(host(X) - ref).max() <= tol * np.abs(ref).max(), (with_D, solve, tree == units)


@pytest.mark.parametrize("kind", ["grid2d", "grid3d"])
@pytest.mark.parametrize("r", [1, 2, 16])
def test_inner_cg(gpu, kind, r):
    """Embedding through the inner CG (r = 1 in the elimination form too)."""
    import torch
    g = _graph(kind)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    off = np.flatnonzero(ot.in_tree == 0)
    add = off[::61]
    in_s = ot.in_tree.copy()
    in_s[add] = 1
    h0 = rng.gaussian_block(11, 3, g.n, r)
    ref, _ = oracle.heat(og, in_s, oracle.embed(og, ot, in_s, h0, 2, 1e-13, 3000))
    with _both(gpu, g) as (ctx, units, rounds):
        for tree in (rounds, units):
            S = gpu.grass_sparsifier_create(ctx, tree)
            try:
                gpu.grass_sparsifier_add(ctx, S, dev(add.astype(np.int64)))
                heat = torch.empty(ref.shape[0], dtype=torch.float64, device="cuda")
                for scan in (1, 0) if r == 1 else (1,):
                    gpu.grass_ctx_set_param(ctx, "euler_solve", scan)
                    gpu.grass_embed(ctx, S, dev(h0), r, 2, gpu.GRASS_FP64, 1e-13, 3000, None, heat)
                    assert np.abs(host(heat) - ref).max() <= 1e-10 * ref.max(), (tree == units, scan)
            finally:
                gpu.grass_sparsifier_destroy(S)


@pytest.mark.parametrize("kind", ["grid2d", "grid3d"])
@pytest.mark.parametrize("inner", [0, 1, 50])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pcg(gpu, kind, inner, prec):
    """The tree alone (0), one inner step in closed form (1), the inner CG (50)."""
    import torch
    g = _graph(kind)
    og = oracle.from_graph(g)
    ot = oracle.build_tree(og)
    add = np.flatnonzero(ot.in_tree == 0)[::9].astype(np.int64)
    b = rng.normal(1, rng.STREAM_RHS, g.n)
    A = sp.csr_matrix((g.val, g.col, g.rowptr), shape=(g.n, g.n))
    P, tol = (gpu.GRASS_FP64, 1e-6) if prec == "fp64" else (gpu.GRASS_FP32, 1e-8)
    with _both(gpu, g) as (ctx, units, rounds):
        for tree in (rounds, units):
            S = gpu.grass_sparsifier_create(ctx, tree)
            try:
                gpu.grass_sparsifier_add(ctx, S, dev(add))
                x = torch.zeros(g.n, dtype=torch.float64, device="cuda")
                status, st = gpu.grass_pcg_solve(ctx, S, dev(b), x, tol, 5000, P, 1e-3, 1e-8, inner)
                assert status == gpu.GRASS_OK
                assert np.linalg.norm(b - A @ host(x)) <= tol * np.linalg.norm(b)
            finally:
                gpu.grass_sparsifier_destroy(S)
