"""FP64 solves with the folded factor (G = L21 L11^-1 P) against a dense solve, at the edges of
their tiles: panel widths below, at and above 64, fronts of one row to several 128-row tiles,
right-hand-side counts around the 8 columns of an item, both launch modes."""
import numpy as np
import pytest
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, laplacian_1d, random_sparse_pencil

pytestmark = pytest.mark.gpu

PENCILS = {
    "one_row": (lambda: laplacian_1d(1), False),
    "path_65": (lambda: laplacian_1d(65, mass=True), False),
    "dense_64": (lambda: random_sparse_pencil(64, 0.9, 1), True),
    "dense_65": (lambda: random_sparse_pencil(65, 0.9, 2), True),
    "dense_323": (lambda: random_sparse_pencil(323, 0.5, 3), True),
    "gauss_432": (lambda: gaussian_pencil((6, 6, 3), seed=4), False),
}


@pytest.mark.parametrize("mode", ["sweep", "per_step"])
@pytest.mark.parametrize("name", sorted(PENCILS))
def test_solve_matches_dense(gpu_lib, name, mode):
    make, dense = PENCILS[name]
    p = make()
    ctx = gpu_lib.Context(0)
    ctx.set_solve_mode(mode)
    sym = ctx.analyze(p.rowptr, p.colind, dense=dense)
    a = torch.tensor(p.a, device="cuda")
    b = torch.tensor(p.b, device="cuda")
    sigma = 0.37
    f = sym.factor(a, b, [sigma], "fp64")
    M = p.dense("a") - sigma * p.dense("b")
    # backward error of the LDL^T solve: n u |L| |D| |L^T|, the growth bounded by max|L|
    tol = 16 * p.n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1])
    for k in (1, 2, 3, 4, 5, 7, 8, 9, 17, 33):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
        ref = np.linalg.solve(M, R)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


BLOCK = {
    "dense_700": (lambda: random_sparse_pencil(700, 0.5, 6), True, (190, 256, 300)),
    "dense_513": (lambda: random_sparse_pencil(513, 0.6, 7), True, (250, 257)),
    "gauss_864": (lambda: gaussian_pencil((6, 6, 6), seed=4), False, (190, 193, 320)),
    "gauss_2000": (lambda: gaussian_pencil((10, 10, 10), (0.3, 2.0), seed=5), False, (64, 65, 128)),
}


def block_case(gpu_lib, name, mode):
    make, dense, ks = BLOCK[name]
    p = make()
    ctx = gpu_lib.Context(0)
    ctx.set_gemm_mode(mode)
    sym = ctx.analyze(p.rowptr, p.colind, dense=dense)
    f = sym.factor(torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda"), [-0.83], "fp64")
    M = p.dense("a") + 0.83 * p.dense("b")
    tol = 16 * p.n * 1.1e-16 * np.linalg.cond(M) * max(1.0, f.stats(0)[1])
    return f, M, tol, ks


@pytest.mark.parametrize("mode", ["tensor", "simt"])
@pytest.mark.parametrize("name", sorted(BLOCK))
def test_block_solve_matches_dense(gpu_lib, name, mode):
    # sizes that take the tensor-core sweeps in "tensor" mode, right-hand sides around the 64 and
    # 128 of an item
    f, M, tol, ks = block_case(gpu_lib, name, mode)
    for k in ks:
        R = np.random.default_rng(k).standard_normal((M.shape[0], k))
        X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
        ref = np.linalg.solve(M, R)
        assert np.linalg.norm(X - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("mode", ["tensor", "simt"])
def test_block_solve_column_scales(gpu_lib, mode):
    # every right-hand-side column keeps its own scale: factors of 2^+-300 and 2^-960, a zero
    # column, and non-finite entries that reach their own column only
    f, M, tol, _ = block_case(gpu_lib, "gauss_864", mode)
    k = 192
    R = np.random.default_rng(9).standard_normal((M.shape[0], k))
    scale = np.ones(k)
    scale[[3, 70]], scale[[4, 140]], scale[[5, 150]] = 2.0 ** 300, 2.0 ** -300, 2.0 ** -960
    R = R * scale
    R[:, 6] = 0.0
    bad = {7: np.inf, 130: np.nan}
    for c, v in bad.items():
        R[M.shape[0] // 2, c] = v
    X = f.solve(0, torch.tensor(R, device="cuda"), refine=0).cpu().numpy()
    good = [c for c in range(k) if c not in bad and c != 6]
    ref = np.linalg.solve(M, R[:, good] / scale[good])
    err = np.linalg.norm(X[:, good] / scale[good] - ref, axis=0)
    assert (err <= tol * np.linalg.norm(ref, axis=0)).all()
    assert (X[:, 6] == 0.0).all()
    for c in bad:
        assert not np.isfinite(X[:, c]).any() or np.isnan(X[:, c]).any()


def test_half_solve_matches_lanczos_frame(gpu_lib):
    # the DOS estimate starts from x0 = G^-T y0 (B = G G^T): ||x0||_B = ||y0||, so the first
    # Lanczos vector's Ritz weights sum to one and a 1-step run returns y0^T G^-1 A G^-T y0 / y0^T y0
    p = gaussian_pencil((5, 4, 3), seed=7)
    ctx, sym, a, b = setup(gpu_lib, p)
    y = torch.randn(p.n, 4, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    runs = sym.dos_estimate(a, b, p.n // 2, y)
    lam = np.linalg.eigvals(np.linalg.solve(p.dense("b"), p.dense("a"))).real
    for th, z2 in runs:
        assert abs(z2.sum() - 1.0) <= 1e-10
        assert th.min() >= lam.min() - 1e-8 * abs(lam).max() and th.max() <= lam.max() + 1e-8 * abs(lam).max()
