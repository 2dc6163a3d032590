"""The Rayleigh-Ritz eigensolver through the Lanczos runs that use it: orders of 1 to several blocks,
odd and even, one to sixteen runs solved together, against the oracle's tridiagonal eigenvalues and
weights, and a run that ends early among longer ones."""
import numpy as np
import pytest
import torch

from oracle import dos
from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, laplacian_1d, normal_block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps,nv", [(1, 2), (2, 4), (3, 16), (33, 8), (96, 2), (97, 4), (128, 1), (150, 2)])
def test_runs_match_oracle(gpu_lib, steps, nv):
    p = gaussian_pencil((5, 5, 5), seed=3)
    ctx, sym, a, b = setup(gpu_lib, p)
    X0 = normal_block(p.n, nv, steps)
    runs = sym.dos_lanczos(a, b, steps, torch.tensor(X0, device="cuda"))
    A, B = p.dense("a"), p.dense("b")
    for c in range(nv):
        th_o, z_o, _, _ = dos.lanczos_ritz(A, B, X0[:, c], steps)
        th, z = runs[c]
        assert th.size == th_o.size
        assert np.abs(th - th_o).max() <= 1e-8 * np.abs(th_o).max()
        assert np.abs(z - z_o).max() <= 1e-8
        assert abs(z.sum() - 1.0) <= 1e-10


def test_early_end_among_full_runs(gpu_lib):
    # a start vector in the span of 5 eigenvectors ends its run after 5 steps
    n, steps = 200, 20
    p = laplacian_1d(n)
    ctx, sym, a, b = setup(gpu_lib, p)
    j = np.arange(1, n + 1)
    V = np.sqrt(2.0 / (n + 1)) * np.sin(np.pi * np.outer(j, [3, 50, 90, 130, 180]) / (n + 1))
    X0 = normal_block(n, 4, 1)
    X0[:, 2] = V @ np.array([1.0, 2.0, -1.0, 0.5, 1.5])
    runs = sym.dos_lanczos(a, b, steps, torch.tensor(X0, device="cuda"))
    assert [r[0].size for r in runs] == [steps, steps, 5, steps]
    lam = 2.0 - 2.0 * np.cos(np.pi * np.array([3, 50, 90, 130, 180]) / (n + 1))
    assert np.abs(runs[2][0] - np.sort(lam)).max() <= 1e-10
