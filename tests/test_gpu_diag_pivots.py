"""The diagonal-block kernel's pivots against Bunch-Kaufman in NumPy on one block: the number of 2x2
pivots and the largest entry of L, on matrices where the diagonal passes, where another row's
diagonal is swapped in, where the second search keeps the diagonal, and where 2x2 pivots are due."""
import numpy as np
import pytest
import torch

from workloads.pencils import Pencil

pytestmark = pytest.mark.gpu
ALPHA = (1.0 + np.sqrt(17.0)) / 8.0


def bunch_kaufman(A):
    A = A.copy()
    n = A.shape[0]
    lmax, n2, kept, swapped = 0.0, 0, 0, 0
    k = 0
    while k < n:
        two, r = False, k
        if k + 1 < n:
            r = k + 1 + int(np.argmax(np.abs(A[k + 1:, k])))
            lam = abs(A[r, k])
            if abs(A[k, k]) < ALPHA * lam:
                row = np.abs(A[r, k:].copy())
                row[r - k] = 0.0
                sig = row.max()
                if abs(A[k, k]) * sig >= ALPHA * lam * lam:
                    kept, r = kept + 1, k
                elif abs(A[r, r]) >= ALPHA * sig:
                    swapped += 1
                else:
                    two = True
            else:
                r = k
        s = k + 1 if two else k
        A[[s, r]] = A[[r, s]]
        A[:, [s, r]] = A[:, [r, s]]
        w = 2 if two else 1
        if k + w < n:
            L = np.linalg.solve(A[k:k + w, k:k + w], A[k:k + w, k + w:]).T
            lmax = max(lmax, np.abs(L).max())
            A[k + w:, k + w:] -= L @ A[k:k + w, k + w:]
        n2, k = n2 + two, k + w
    return lmax, n2, kept, swapped


@pytest.mark.parametrize("diag", [0.0, 0.3, 1.0, 6.0, 30.0])
@pytest.mark.parametrize("n", [2, 31, 33, 64])
def test_pivots_match_numpy(gpu_lib, n, diag):
    rng = np.random.default_rng(int(17 * n + diag * 10))
    A = rng.standard_normal((n, n))
    A = np.tril(A, -1) + np.tril(A, -1).T + np.diag(diag * rng.standard_normal(n))
    p = Pencil(n, np.arange(0, n * n + 1, n, dtype=np.int64), np.tile(np.arange(n, dtype=np.int32), n),
               A.ravel().copy(), np.eye(n).ravel().copy())
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind, dense=True)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [0.0], "fp64")
    lmax, n2, kept, swapped = bunch_kaufman(A)
    _, got_lmax, got_n2 = f.stats(0)
    assert got_n2 == n2
    # rounding differs along the elimination: n u growth^2
    assert abs(got_lmax - lmax) <= 1e-9 * lmax
    if n == 64 and diag == 1.0:
        assert n2 > 0 and kept + swapped > 0
