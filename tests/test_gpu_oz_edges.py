"""Tensor-core products at the edges of the pipelined kernel: row tiles without entries or with one
piece, pieces with one and with thousands of entries, groups of 16 pieces just full and just begun,
and ragged output columns, against numpy in the bound the split guarantees."""
import numpy as np
import pytest
import torch

from workloads.pencils import Pencil

pytestmark = pytest.mark.gpu


def band_pencil(n, reach, dense_rows, seed):
    """Diagonal, a few entries within `reach`, and `dense_rows` full rows / columns."""
    rng = np.random.default_rng(seed)
    cols = [set() for _ in range(n)]
    for i in range(n):
        cols[i].add(i)
        for j in rng.integers(max(0, i - reach), min(n, i + reach + 1), size=3):
            cols[i].add(int(j))
            cols[int(j)].add(i)
    for d in dense_rows:
        for j in range(n):
            cols[d].add(j)
            cols[j].add(d)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum([len(c) for c in cols])
    colind = np.concatenate([np.sort(np.fromiter(c, dtype=np.int32)) for c in cols])
    a = rng.standard_normal(colind.size) * 2.0 ** rng.integers(-40, 40, size=colind.size)
    return Pencil(n, rowptr, colind, a, rng.standard_normal(colind.size))


@pytest.mark.parametrize("dense_rows", [(), (5,), tuple(range(300, 430))])
@pytest.mark.parametrize("n,reach,k", [(2048, 1, 48), (2049, 40, 63), (2500, 600, 65), (3001, 1500, 130)])
def test_sparse_product(gpu_lib, n, reach, k, dense_rows):
    p = band_pencil(n, reach, dense_rows, n)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    X = np.random.default_rng(k).standard_normal((n, k))
    a = p.a.copy()
    a[p.rowptr[130]:p.rowptr[131]] = 0.0           # a row of zeros
    Y = sym.spmm(torch.tensor(a, device="cuda"), torch.tensor(p.b, device="cuda"), torch.tensor(X, device="cuda"),
                 1.0, -0.25).cpu().numpy()
    A, B = np.zeros((n, n)), np.zeros((n, n))
    A[p.rows(), p.colind], B[p.rows(), p.colind] = a, p.b
    m = np.diff(p.rowptr)[:, None]
    xm = np.abs(X).max(axis=0)[None, :]
    bound = 8 * 2.0 ** -53 * m * (np.abs(A).max(axis=1)[:, None] + np.abs(B).max(axis=1)[:, None]) * xm
    bound += 2.0 ** -52 * (m + 2) * (np.abs(A) @ np.abs(X) + np.abs(B) @ np.abs(X))
    assert (np.abs(Y - (A @ X - 0.25 * (B @ X))) <= bound).all()


@pytest.mark.parametrize("n,k1,k2", [(2048, 48, 48), (2079, 64, 129), (16 * 32 * 9, 65, 191), (16 * 32 * 9 + 1, 128, 64)])
def test_dense_products(gpu_lib, n, k1, k2):
    ctx = gpu_lib.Context(0)
    rng = np.random.default_rng(n + k1)
    X, Y, Q = rng.standard_normal((n, k1)), rng.standard_normal((n, k2)), rng.standard_normal((k1, k2))
    Xd, Yd = torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda")
    G = ctx.dense_gram(Xd, Yd).cpu().numpy()
    bound = 8 * 2.0 ** -53 * n * np.abs(X).max(axis=0)[:, None] * np.abs(Y).max(axis=0)[None, :]
    assert (np.abs(G - X.T @ Y) <= bound + 2.0 ** -52 * n * (np.abs(X).T @ np.abs(Y))).all()
    Z = ctx.dense_gemm(Xd, torch.tensor(Q, device="cuda"), torch.empty(n, k2, dtype=torch.float64, device="cuda"))
    bound = 8 * 2.0 ** -53 * k1 * np.abs(X).max(axis=1)[:, None] * np.abs(Q).max(axis=0)[None, :]
    assert (np.abs(Z.cpu().numpy() - X @ Q) <= bound + 2.0 ** -52 * k1 * (np.abs(X) @ np.abs(Q))).all()
