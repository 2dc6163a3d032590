"""Lanczos density-of-states runs of 1 to 256 vectors against their defining property: the Ritz
values and weights of m steps integrate the first 2 m - 1 moments of the start vector's spectral
measure of B^-1 A exactly.  Sizes around the 32 entries, 8 warps and 2,048-entry chunks of the
re-orthogonalisation, runs shorter and longer than 8 vectors."""
import numpy as np
import pytest
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [1, 2, 16, 32, 64, 256])
@pytest.mark.parametrize("dims,steps", [((3, 3, 3), 3), ((5, 4, 3), 9), ((8, 7, 6), 20)])
def test_moments(gpu_lib, dims, steps, nv):
    p = gaussian_pencil(dims, (0.3, 2.0), seed=21)
    ctx, sym, a, b = setup(gpu_lib, p)
    x0 = np.random.default_rng(nv).standard_normal((p.n, nv))
    runs = sym.dos_lanczos(a, b, steps, torch.tensor(x0, device="cuda"))
    A, B = p.dense("a"), p.dense("b")
    L = np.linalg.cholesky(B)
    C = np.linalg.solve(L, np.linalg.solve(L, A).T)      # L^-1 A L^-T
    y = L.T @ x0
    y /= np.linalg.norm(y, axis=0)
    rho = np.linalg.norm(C, 2)
    # the recurrence's rounding is n u cond(B) relative to the spectral radius, moment by moment
    tol = 64 * p.n * 1.1e-16 * np.linalg.cond(B)
    v = y.copy()
    for q in range(1, 6):
        v = C @ v
        exact = (y * v).sum(axis=0)
        got = np.array([(z2 * th ** q).sum() for th, z2 in runs])
        assert (np.abs(got - exact) <= q * tol * rho ** q).all()
