"""The returned eigenvalues are the Rayleigh quotients of the returned vectors whatever the scale of the basis
functions: rows and columns of A and B multiplied by 2^-span .. 2^span, vectors before convergence."""
import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("driver", ["subspace", "lanczos"])
@pytest.mark.parametrize("span", [0, 5, 15])
def test_quotients_of_a_scaled_pencil(gpu_lib, span, driver):
    p = gaussian_pencil((6, 5, 6), seed=9)
    S = 2.0 ** np.random.default_rng(span).integers(-span, span + 1, p.n)
    scale = S[p.rows()] * S[p.colind]
    ctx = gpu_lib.Context(0)
    sym = ctx.analyze(p.rowptr, p.colind)
    a, b = torch.tensor(p.a * scale, device="cuda"), torch.tensor(p.b * scale, device="cuda")
    f = sym.factor(a, b, [-0.3141], "fp64", allow_singular=True)
    V0 = torch.tensor(normal_block(p.n, 20, 11), device="cuda")
    kw = dict(max_iter=3, n_expect=21) if driver == "subspace" else dict(max_iter=3, k_out=31, driver="lanczos")
    pr = f.slice_solve(0, -2.0, 1.0, V0, allow_noconv=True, **kw)
    X = pr.X.cpu().numpy().astype(np.longdouble)
    scale = S[:, None] * S[None, :]
    A, B = (p.dense("a") * scale).astype(np.longdouble), (p.dense("b") * scale).astype(np.longdouble)
    num, den = (X * (A @ X)).sum(axis=0), (X * (B @ X)).sum(axis=0)
    size = (np.abs(X) * (np.abs(A) @ np.abs(X))).sum(axis=0) + np.abs(num / den) * (np.abs(X) * (np.abs(B) @ np.abs(X))).sum(axis=0)
    # one rounding of the quotient; rows of A and B to 2^-62 and vectors to 2^-53 of their largest scaled entry,
    # which the residual multiplies; scales that follow S to a factor of 8 (the diagonal of the unscaled pencil)
    resid = np.abs(A @ X - (B @ X) * (num / den))
    big = np.abs(X * S[:, None]).max(axis=0)
    first = 8 * 2 * 2.0 ** -52 * big * (resid / S[:, None]).sum(axis=0)
    tol = 2.0 ** -52 * np.abs(num / den) + (2.0 ** -56 * size + first) / den
    assert (np.abs(pr.theta - num / den) <= tol).all()
