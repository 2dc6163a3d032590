"""FP64 solves of few right-hand sides against a dense solve where levels halve their items: levels
of one tile (halved three times) up to levels of more items than warps (not halved), widths of
every kind of reduction (1, 2, 4 and 8 values, odd counts filled up), one and two chunks of
right-hand sides, 2 x 2 pivots and pivots whose reciprocal has too few bits."""
import dataclasses

import numpy as np
import pytest
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, random_sparse_pencil

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["sweep", "per_step"])
@pytest.mark.parametrize("dims", [(9, 8, 7), (12, 10, 10)])
def test_split_levels_match_dense(gpu_lib, dims, mode):
    p = gaussian_pencil(dims, (0.3, 2.0), seed=11)
    ctx, sym, a, b = setup(gpu_lib, p)
    ctx.set_solve_mode(mode)
    f = sym.factor(a, b, [-1.1], "fp64")
    M = p.dense("a") + 1.1 * p.dense("b")
    # backward error of the LDL^T solve: n u |L| |D| |L^T|, the growth bounded by max|L|
    tol = 16 * p.n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1])
    for k in (1, 2, 3, 5, 6, 7, 8, 11):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
        ref = np.linalg.solve(M, R)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [0, 1004, -1004])
def test_pivot_reciprocals(gpu_lib, scale):
    # D with 2 x 2 blocks; scaled by 2^+-1004 its 1 x 1 pivots leave the range of the reciprocals.
    # The scaled systems keep 1 x 1 pivots (diagonally dominant): a 2 x 2 determinant of theirs
    # would not be finite.
    p = random_sparse_pencil(130, 0.5, 12)
    if scale:
        a = p.a.copy()
        rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
        a[rows == p.colind] += 4.0 * np.abs(p.dense("a")).sum(axis=1).max()
        p = dataclasses.replace(p, a=a)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    M = p.dense("a")
    a = torch.tensor(np.ldexp(p.a, scale), device="cuda")
    f = sym.factor(a, torch.tensor(p.b, device="cuda"), [0.0], "fp64")
    if scale == 0:
        assert f.stats(0)[2] > 0
    tol = 16 * p.n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1])
    for k in (1, 4, 8):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        X = f.solve(0, torch.tensor(np.ldexp(R, scale), device="cuda"), refine=0).cpu().numpy()
        ref = np.linalg.solve(M, R)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)
