"""The band-energy gradient on the tensor cores against numpy: rows ragged to the 128- and 64-row
tiles, column counts around the 32 of a piece and the 16 pieces of a group, one output only, and
non-finite rows, in the bound the digit split guarantees; below its sizes the CUDA cores answer."""
import ctypes as C

import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil

pytestmark = pytest.mark.gpu


def setup_case(gpu_lib, dims, exps, ne, seed):
    p = gaussian_pencil(dims, exps, seed=seed)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((p.n, ne)) * 2.0 ** rng.integers(-20, 20, size=(p.n, 1))
    lam = np.sort(rng.uniform(-40.0, 2.0, ne))
    return p, sym, X, lam


@pytest.mark.parametrize("ne", [47, 48, 49, 64, 511, 512, 513, 700])
def test_gradient_entries(gpu_lib, ne):
    p, sym, X, lam = setup_case(gpu_lib, (9, 11, 11), (0.3, 2.0), ne, 3)     # N = 2,178
    ga, gb = sym.band_energy_grad(torch.tensor(X, device="cuda"), torch.tensor(lam, device="cuda"))
    r, c = p.rows(), p.colind
    a, b = (X @ X.T)[r, c], -((X * lam) @ X.T)[r, c]
    xm, lm = np.abs(X).max(axis=1), np.abs(X * lam).max(axis=1)
    split = 8 * 2.0 ** -53 * ne
    own = 2.0 ** -52 * (ne + 2)
    assert (np.abs(ga.cpu().numpy() - a) <= split * xm[r] * xm[c] + own * (np.abs(X) @ np.abs(X).T)[r, c]).all()
    tol_b = split * np.maximum(xm[r] * lm[c], lm[r] * xm[c]) + own * (np.abs(X * lam) @ np.abs(X).T)[r, c]
    assert (np.abs(gb.cpu().numpy() - b) <= tol_b).all()


def test_one_output_and_non_finite_rows(gpu_lib):
    p, sym, X, lam = setup_case(gpu_lib, (9, 11, 11), (0.3, 2.0), 96, 4)
    X[1000, 5], X[70, 90] = np.inf, np.nan
    Xd, ld = torch.tensor(X, device="cuda"), torch.tensor(lam, device="cuda")
    ga = torch.full((p.nnz,), 7.0, dtype=torch.float64, device="cuda")
    rc = sym.ctx.lib.ss_band_energy_grad(sym.h, C.c_void_p(Xd.data_ptr()), C.c_void_p(ld.data_ptr()), 96,
                                         C.c_void_p(ga.data_ptr()), None)
    sym.ctx.check(rc, "ss_band_energy_grad")
    g = ga.cpu().numpy()
    r, c = p.rows(), p.colind
    bad = np.isin(r, (70, 1000)) | np.isin(c, (70, 1000))
    assert not np.isfinite(g[bad]).any() and np.isfinite(g[~bad]).all()
