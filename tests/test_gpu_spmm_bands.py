"""CUDA-core sparse products over bands: rows that end at, before and after a multiple of the 32 lanes and of the
unrolled trips, every chunk width, few and many rows (both forms of the product), and an infinity in the block
that reaches only the rows it belongs to."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def band(n, h):
    r = np.repeat(np.arange(n), 2 * h + 1)
    c = r + np.tile(np.arange(-h, h + 1), n)
    keep = (c >= 0) & (c < n)
    return r[keep], c[keep]


@pytest.mark.parametrize("n", [300, 5000])
@pytest.mark.parametrize("h", [0, 15, 16, 32, 48, 64])
def test_band_products(gpu_lib, n, h):
    r, c = band(n, h)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    rng = np.random.default_rng(h)
    av, bv = rng.standard_normal(r.size), rng.standard_normal(r.size)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(rowptr, c.astype(np.int32))
    a, b = torch.tensor(av, device="cuda"), torch.tensor(bv, device="cuda")

    def product(v, X):
        out = np.zeros_like(X)
        np.add.at(out, r, v[:, None] * X[c])
        return out

    for k in (1, 3, 5, 6, 7, 8, 15, 16, 20, 25, 31, 33, 42, 47):
        X = rng.standard_normal((n, k))
        Xd = torch.tensor(X, device="cuda")
        al, be = np.linspace(0.5, 2.0, k), np.linspace(-1.0, 0.25, k)
        ax, bx = product(av, X), product(bv, X)
        bound_a, bound_b = product(np.abs(av), np.abs(X)), product(np.abs(bv), np.abs(X))
        # error of a sum of m terms in any order: m u of the sum of magnitudes
        m, u = 2 * h + 1, 1.2e-16
        Y = sym.spmm(a, b, Xd).cpu().numpy()
        assert (np.abs(Y - ax) <= 2 * (m + 2) * u * bound_a).all()
        Y = sym.spmm(a, b, Xd, al, be).cpu().numpy()
        assert (np.abs(Y - ax * al - bx * be) <= 2 * (m + 6) * u * (bound_a * al + bound_b * np.abs(be))).all()
    X[n // 2, 0] = np.inf
    Y = sym.spmm(a, b, torch.tensor(X, device="cuda")).cpu().numpy()
    touched = np.zeros(n, bool)
    touched[r[c == n // 2]] = True
    assert not np.isfinite(Y[touched, 0]).any() and np.isfinite(Y[~touched, 0]).all() and np.isfinite(Y[:, 1:]).all()
