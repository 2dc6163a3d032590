"""The band-energy gradient takes the tensor cores only where the pattern fills their tiles: short rows and
scattered entries stay on the CUDA cores, blocks of neighbours leave them, with the same entries either way."""
import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil

pytestmark = pytest.mark.gpu


def band(n, h):
    r = np.repeat(np.arange(n), 2 * h + 1)
    c = r + np.tile(np.arange(-h, h + 1), n)
    keep = (c >= 0) & (c < n)
    return r[keep], c[keep]


def scattered(n, d):
    rng = np.random.default_rng(1)
    r, c = rng.integers(0, n, n * d // 2), rng.integers(0, n, n * d // 2)
    key = np.unique(np.concatenate([r * n + c, c * n + r, np.arange(n) * (n + 1)]))
    return key // n, key % n


PATTERNS = {"band_1": (lambda: band(3000, 1), 96, False), "band_4": (lambda: band(3000, 4), 300, False),
            "scattered_20": (lambda: scattered(3000, 20), 300, False), "band_64": (lambda: band(3000, 64), 300, True),
            "gauss_2178": (lambda: (lambda p: (p.rows(), p.colind))(gaussian_pencil((9, 11, 11), (0.3, 2.0), seed=3)),
                           48, True)}


@pytest.mark.parametrize("name", sorted(PATTERNS))
def test_route_and_entries(gpu_lib, name):
    make, ne, tensor = PATTERNS[name]
    r, c = make()
    n = int(r.max()) + 1
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(rowptr, c.astype(np.int32))
    rng = np.random.default_rng(2)
    X, lam = rng.standard_normal((n, ne)), np.sort(rng.uniform(-4.0, 2.0, ne))
    ctx.profile(["sddmm"])
    ga, gb = sym.band_energy_grad(torch.tensor(X, device="cuda"), torch.tensor(lam, device="cuda"))
    ctx.profile_query("sddmm")
    assert (ctx.profile_query_tensor("sddmm") > 0.0) == tensor
    ctx.profile()
    a, b = (X[r] * X[c]).sum(1), -(X[r] * lam * X[c]).sum(1)
    xm = np.abs(X).max()
    tol = (8 * 2.0 ** -53 * ne + 2.0 ** -52 * (ne + 2) * ne) * xm * xm
    assert np.abs(ga.cpu().numpy() - a).max() <= tol
    assert np.abs(gb.cpu().numpy() - b).max() <= 4.0 * tol
