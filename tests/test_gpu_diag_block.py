"""The diagonal-block and panel kernels at the edges of their sizes: panel widths of 1 to 65
columns, blocks that need symmetric swaps and 2x2 pivots in every place (zero diagonals, also
across the 16-column quarters), and a zero matrix row; inertia against
the eigenvalues and solves against a dense solve."""
import numpy as np
import pytest
import torch

from workloads.pencils import Pencil

pytestmark = pytest.mark.gpu


def dense_pencil(A):
    n = A.shape[0]
    rowptr = np.arange(0, n * n + 1, n, dtype=np.int64)
    colind = np.tile(np.arange(n, dtype=np.int32), n)
    return Pencil(n, rowptr, colind, A.ravel().copy(), np.eye(n).ravel().copy())


def symmetric(n, seed, zero_diag):
    A = np.random.default_rng(seed).standard_normal((n, n))
    A = A + A.T
    if zero_diag:
        A[np.arange(n), np.arange(n)] = 0.0
    return A


@pytest.mark.parametrize("zero_diag", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 97, 130, 200])
def test_inertia_and_solve(gpu_lib, n, zero_diag):
    A = symmetric(n, 100 + n, zero_diag and n > 1)
    p = dense_pencil(A)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    a, b = torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda")
    f = sym.factor(a, b, [0.0], "fp64")
    neg, zero, pos, tiny = f.inertia(0)
    lam = np.linalg.eigvalsh(A)
    assert (neg, zero, pos, tiny) == (int((lam < 0).sum()), 0, int((lam > 0).sum()), False)
    R = np.random.default_rng(n).standard_normal((n, 3))
    X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
    ref = np.linalg.solve(A, R)
    tol = 16 * n * 1.1e-16 * np.linalg.cond(A) * max(1.0, f.stats(0)[1]) ** 2
    assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


def test_two_by_two_pivot_in_every_place(gpu_lib):
    # blocks [[0, 1], [1, 0]] on the diagonal after one leading 1x1 pivot: 2x2 pivots at columns
    # 1, 3, .., also across the quarters (15, 16), (31, 32), (47, 48)
    n = 64
    A = np.zeros((n, n))
    A[0, 0] = 3.0
    for i in range(1, n - 1, 2):
        A[i, i + 1] = A[i + 1, i] = 2.0
    A[n - 1, n - 1] = -1.0
    B = np.random.default_rng(5).standard_normal((90, n)) * 0.1
    M = np.block([[A, B.T], [B, 4.0 * np.eye(90)]])
    p = dense_pencil(M)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    a, b = torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda")
    f = sym.factor(a, b, [0.0], "fp64")
    lam = np.linalg.eigvalsh(M)
    assert f.inertia(0)[:3] == (int((lam < 0).sum()), 0, int((lam > 0).sum()))
    perm_ok = np.sort(sym.perm())
    assert np.array_equal(perm_ok, np.arange(M.shape[0]))
    R = np.random.default_rng(1).standard_normal((M.shape[0], 2))
    X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
    tol = 16 * n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1]) ** 2
    ref = np.linalg.solve(M, R)
    assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


def test_zero_row_is_counted(gpu_lib):
    n = 20
    A = symmetric(n, 3, False)
    A[7, :] = A[:, 7] = 0.0
    p = dense_pencil(A)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [0.0], "fp64",
                   allow_singular=True)
    lam = np.linalg.eigvalsh(np.delete(np.delete(A, 7, 0), 7, 1))
    assert f.singular and f.inertia(0)[:3] == (int((lam < 0).sum()), 1, int((lam > 0).sum()))
