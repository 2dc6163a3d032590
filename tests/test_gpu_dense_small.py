"""Gram matrices and tall products of few columns (CUDA cores) against NumPy at the edges of their
tiles: columns around 16 and 32, rows around 32 and 64, every number of rows a block, strides wider
than the matrix, alpha, beta and the transposed factor."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 1.1e-16


def wide(rng, n, k):
    t = torch.tensor(rng.standard_normal((n, k + 3)), device="cuda")
    return t[:, :k]


@pytest.mark.parametrize("n", [1, 31, 33, 65, 700, 5000, 40000])
@pytest.mark.parametrize("k1,k2", [(1, 1), (15, 16), (16, 17), (17, 31), (32, 33), (33, 47), (47, 40)])
def test_small_products_match_numpy(gpu_lib, n, k1, k2):
    rng = np.random.default_rng(1000 * k1 + n)
    ctx = gpu_lib.Context(0)
    X, Y = wide(rng, n, k1), wide(rng, n, k2)
    x, y = X.cpu().numpy(), Y.cpu().numpy()
    # a sum of n products in any order: (n + 2) u |x|^T |y|
    G = ctx.dense_gram(X, Y).cpu().numpy()
    assert (np.abs(G - x.T @ y) <= 2 * (n + 2) * U * (np.abs(x).T @ np.abs(y))).all()
    for transq in (False, True):
        q = rng.standard_normal((k2, k1) if transq else (k1, k2))
        Z = wide(rng, n, k2)
        z = Z.cpu().numpy()
        qq = q.T if transq else q
        ctx.dense_gemm(X, torch.tensor(q, device="cuda"), Z, alpha=-1.5, beta=0.5, transq=transq)
        bound = 2 * (k1 + 4) * U * (1.5 * np.abs(x) @ np.abs(qq) + 0.5 * np.abs(z))
        assert (np.abs(Z.cpu().numpy() - (0.5 * z - 1.5 * x @ qq)) <= bound).all()
