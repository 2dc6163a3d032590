"""CUDA-core sparse products of few columns against numpy: every chunk width (1 .. 8 columns, one
to six chunks), with and without the B term and the column factors, rows of 1 to 3 entries (few
lanes busy) and long rows."""
import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil, laplacian_1d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["path", "gauss"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 15, 16, 17, 23, 31, 33, 41, 47])
def test_thin_products(gpu_lib, name, k):
    p = laplacian_1d(130, mass=True) if name == "path" else gaussian_pencil((5, 4, 5), seed=2)
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    a, b = torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda")
    X = np.random.default_rng(k).standard_normal((p.n, k))
    Xd = torch.tensor(X, device="cuda")
    A, B = p.dense("a"), p.dense("b")
    al, be = np.linspace(0.5, 2.0, k), np.linspace(-1.0, 0.25, k)
    # error of a sum of m terms in any order: m u of the sum of magnitudes
    m = int(np.diff(p.rowptr).max())
    bound_a, bound_b = np.abs(A) @ np.abs(X), np.abs(B) @ np.abs(X)
    u = 1.2e-16
    Y = sym.spmm(a, b, Xd).cpu().numpy()
    assert (np.abs(Y - A @ X) <= 2 * (m + 2) * u * bound_a).all()
    Y = sym.spmm(a, b, Xd, al).cpu().numpy()
    assert (np.abs(Y - (A @ X) * al) <= 2 * (m + 4) * u * bound_a * al).all()
    Y = sym.spmm(a, b, Xd, al, be).cpu().numpy()
    assert (np.abs(Y - (A @ X) * al - (B @ X) * be) <= 2 * (m + 6) * u * (bound_a * al + bound_b * np.abs(be))).all()
