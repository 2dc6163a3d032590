"""Cholesky-QR of a probe's basis at the edges of the 32-wide panels of its factor: the returned
vectors are B-orthonormal for basis widths of 1 to several panels, and a rank-deficient start
block is reported or recovered, never returned as a basis."""
import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu


def probe(gpu_lib, V0, p):
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.4321], "fp64")
    return f.slice_solve(0, -2.0, 1.0, torch.tensor(V0, device="cuda"), max_iter=2, n_expect=V0.shape[1] + 1,
                         allow_noconv=True)


@pytest.mark.parametrize("k", [1, 2, 31, 32, 33, 64, 65, 95, 97, 160, 303])
def test_basis_is_b_orthonormal(gpu_lib, k):
    p = gaussian_pencil((5, 5, 5), seed=12)
    X = probe(gpu_lib, normal_block(p.n, k, k), p).X.cpu().numpy()
    E = X.T @ p.dense("b") @ X - np.eye(k)
    # two Cholesky-QR passes: a few u times k, times |X|^T |B| |X| (B is nearly singular)
    size = (np.abs(X).T @ np.abs(p.dense("b")) @ np.abs(X)).max()
    assert np.abs(E).max() <= 64 * k * 1.1e-16 * max(1.0, size)


def test_rank_deficient_start_block(gpu_lib):
    p = gaussian_pencil((5, 5, 5), seed=12)
    V0 = normal_block(p.n, 70, 5)
    V0[:, 40] = V0[:, 3]
    try:
        X = probe(gpu_lib, V0, p).X.cpu().numpy()
    except gpu_lib.SisliceError as e:
        assert e.status == gpu_lib.L.SS_ERR_NOCONV
        return
    assert np.abs(X.T @ p.dense("b") @ X - np.eye(70)).max() <= 1e-8
