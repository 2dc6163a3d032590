"""FP64 block solves on the tensor cores, each case shown to have run there by the tensor-core work that the
library counts for it, against a dense solve."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from workloads.pencils import gaussian_pencil, laplacian_1d, random_sparse_pencil

pytestmark = pytest.mark.gpu

PENCILS = {
    # one front of 8 panels of 64 and one of a single row: remainders of one row in every tile column
    "dense_513": (lambda: random_sparse_pencil(513, 0.6, 7), True),
    # one front of 32 panels: enough entries a level for items of 64 right-hand sides
    "dense_2000": (lambda: random_sparse_pencil(2000, 0.2, 8), True),
    "gauss_1728": (lambda: gaussian_pencil((6, 8, 9), seed=5), False),
}
_FACTORS = {}


def factored(gpu_lib, name):
    if name not in _FACTORS:
        make, dense = PENCILS[name]
        p = make()
        ctx = gpu_lib.Context(0)
        sym = ctx.analyze(p.rowptr, p.colind, dense=dense)
        f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.83], "fp64")
        M = p.dense("a") + 0.83 * p.dense("b")
        # backward error of the LDL^T solve: n u |L| |D| |L^T|, the growth bounded by max|L|
        _FACTORS[name] = f, M, 16 * p.n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1])
    return _FACTORS[name]


def solved(f, R, mode="tensor"):
    """X, and the tensor-core flops of the sweeps"""
    f.ctx.set_gemm_mode(mode)
    f.ctx.profile(["solve"])
    X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
    flops = f.ctx.profile_query_tensor("solve")
    f.ctx.profile()
    return X, flops


@pytest.mark.parametrize("name,ks", [("dense_513", (300, 319, 320, 321)), ("gauss_1728", (127, 128, 129, 193, 256)),
                                     ("dense_2000", (63, 64, 65, 96, 97, 127, 128, 129))])
def test_edges_of_the_right_hand_side_tiles(gpu_lib, name, ks):
    f, M, tol = factored(gpu_lib, name)
    n = M.shape[0]
    for k in ks:
        R = np.random.default_rng(k).standard_normal((n, k))
        X, flops = solved(f, R)
        # 28 products of 8-bit digits, at least, to each FP64 product of the two sweeps
        assert flops >= 28 * 4.0 * f.sym.info["l_offdiag_entries"] * k
        ref = np.linalg.solve(M, R)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


def test_few_right_hand_sides(gpu_lib):
    # a warp's 32 right-hand sides and one more, by the residual: a backward error of n u |L| |D| |L^T|
    p = gaussian_pencil((12, 12, 12), seed=1)                             # N = 6,912
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.83], "fp64")
    M = sp.csr_matrix((p.a + 0.83 * p.b, p.colind, p.rowptr), shape=(p.n, p.n))
    norm = abs(M).sum(axis=1).max()
    tol = 16 * p.n * 1.1e-16 * max(1.0, f.stats(0)[1])
    for k in (24, 31, 32, 33):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        X, flops = solved(f, R)
        assert flops >= 28 * 4.0 * sym.info["l_offdiag_entries"] * k
        res = np.linalg.norm(R - M @ X, axis=0)
        assert (res <= tol * (norm * np.linalg.norm(X, axis=0) + np.linalg.norm(R, axis=0))).all()


def test_tiles_of_a_row_or_two(gpu_lib):
    # a path: most panels have one or two rows below them, so whole items of the CUDA cores count, not entries
    p = laplacian_1d(5000, mass=True)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.83], "fp64")
    M = sp.csr_matrix((p.a + 0.83 * p.b, p.colind, p.rowptr), shape=(p.n, p.n))
    norm = abs(M).sum(axis=1).max()
    tol = 16 * p.n * 1.1e-16 * max(1.0, f.stats(0)[1])
    for k in (111, 128, 129, 200):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        X, flops = solved(f, R)
        assert flops > 0.0
        res = np.linalg.norm(R - M @ X, axis=0)
        assert (res <= tol * (norm * np.linalg.norm(X, axis=0) + np.linalg.norm(R, axis=0))).all()


def test_cuda_core_solves_count_no_tensor_work(gpu_lib):
    f, M, _ = factored(gpu_lib, "dense_513")
    assert solved(f, np.ones((M.shape[0], 320)), "simt")[1] == 0.0
    assert solved(f, np.ones((M.shape[0], 8)))[1] == 0.0


@pytest.mark.parametrize("mode", ["tensor", "simt"])
@pytest.mark.parametrize("span", [0, 5, 10, 20])
def test_scaled_basis_keeps_its_digits(gpu_lib, span, mode):
    # S M S with S = 2^-span .. 2^span per row has the solution S^-1 M^-1 R of the right-hand sides S R: a
    # positive definite M, which every pivot order factors stably, solved to its own n u cond(M), not to
    # that of the scaled matrix
    p = random_sparse_pencil(700, 0.5, 6)
    n, k = p.n, 300
    rng = np.random.default_rng(span)
    S = 2.0 ** rng.integers(-span, span + 1, n)
    rows, cols = p.rows(), p.colind
    lam = np.linalg.eigvals(np.linalg.solve(p.dense("b"), p.dense("a"))).real
    sigma = lam.min() - np.ptp(lam)
    ctx = gpu_lib.Context(0)
    ctx.set_schur_mode("simt")                    # the factor itself in plain FP64
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    scale = S[rows] * S[cols]
    # (pivots of 2^-40 of the norm are reported as singular, the factor is there all the same)
    f = sym.factor(torch.tensor(p.a * scale, device="cuda"), torch.tensor(p.b * scale, device="cuda"), [sigma], "fp64",
                   allow_singular=True)
    M = p.dense("a") - sigma * p.dense("b")
    R = rng.standard_normal((n, k))
    X, flops = solved(f, S[:, None] * R, mode)
    assert (flops > 0.0) == (mode == "tensor")
    ref = np.linalg.solve(M, R)
    assert np.linalg.norm(S[:, None] * X - ref) <= 16 * n * 1.1e-16 * np.linalg.cond(M) * np.linalg.norm(ref)


@pytest.mark.parametrize("mode", ["tensor", "simt"])
def test_denormal_right_hand_sides(gpu_lib, mode):
    # whole multiples, up to 2^43, of the smallest denormal: every addition rounds to one of those, n of them
    # to an entry, amplified by cond(M)
    p = random_sparse_pencil(700, 0.5, 6)
    lam = np.linalg.eigvals(np.linalg.solve(p.dense("b"), p.dense("a"))).real
    sigma = lam.min() - np.ptp(lam)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [sigma], "fp64")
    M = p.dense("a") - sigma * p.dense("b")
    k = 300
    N = np.rint(2.0 ** 40 * np.random.default_rng(1).standard_normal((p.n, k)))
    unit = 2.0 ** -1074
    X, flops = solved(f, N * unit, mode)
    assert (flops > 0.0) == (mode == "tensor")
    ref = np.linalg.solve(M, N)
    tol = 16 * p.n * np.linalg.cond(M) * max(1.0, np.linalg.norm(np.linalg.inv(M), 2))
    assert np.abs(X / unit - ref).max() <= tol
