"""The returned eigenvalues are the Rayleigh quotients of the returned vectors, to the last bits:
against quotients summed in extended precision, for column counts around the 64 of a block's tile
and for a row much longer than the rest."""
import numpy as np
import pytest
import torch

from workloads.pencils import Pencil, gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu


def arrow_pencil(n, seed):
    """Tridiagonal plus a full first row and column."""
    rng = np.random.default_rng(seed)
    A = np.zeros((n, n))
    i = np.arange(n)
    A[i, i] = rng.uniform(-1.0, 3.0, n)
    A[i[:-1], i[1:]] = A[i[1:], i[:-1]] = rng.uniform(-1, 1, n - 1)
    A[0, :] = A[:, 0] = 2.0 ** rng.integers(-30, 3, n) * rng.choice([-1.0, 1.0], n)
    r, c = np.nonzero(A)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.add.at(rowptr, r + 1, 1)
    return Pencil(n, np.cumsum(rowptr), c.astype(np.int32), A[r, c], np.where(r == c, 2.0, 0.0))


@pytest.mark.parametrize("name,k", [("gauss", 31), ("gauss", 64), ("gauss", 65), ("arrow", 100)])
def test_quotients(gpu_lib, name, k):
    p = gaussian_pencil((6, 5, 6), seed=9) if name == "gauss" else arrow_pencil(900, 3)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.3141], "fp64")
    V0 = torch.tensor(normal_block(p.n, k, 11), device="cuda")
    pr = f.slice_solve(0, -2.0, 1.0, V0, max_iter=3, n_expect=k + 1, allow_noconv=True)
    X = pr.X.cpu().numpy().astype(np.longdouble)
    A, B = p.dense("a").astype(np.longdouble), p.dense("b").astype(np.longdouble)
    num, den = (X * (A @ X)).sum(axis=0), (X * (B @ X)).sum(axis=0)
    size = (np.abs(X) * (np.abs(A) @ np.abs(X))).sum(axis=0) + np.abs(num / den) * (np.abs(X) * (np.abs(B) @ np.abs(X))).sum(axis=0)
    # one rounding of the quotient, rows of A and B to 2^-62 of their largest entry, the extended sums
    tol = 2.0 ** -52 * np.abs(num / den) + 2.0 ** -56 * size / den
    assert (np.abs(pr.theta - num / den) <= tol).all()
