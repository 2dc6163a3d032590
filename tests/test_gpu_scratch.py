"""What the calls do when scratch memory does not fit, with device allocations made to fail on the host."""
import numpy as np
import pytest
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, laplacian_1d, normal_block

pytestmark = pytest.mark.gpu


def test_gradient_fallback_leaves_the_factors_products(gpu_lib):
    # the lists of the sampled product do not fit: the gradient runs on the CUDA cores, and a factor that
    # used the tensor-core products before goes on using them
    p = gaussian_pencil((8, 8, 9), seed=2)
    ctx, sym, a, b = setup(gpu_lib, p)
    f = sym.factor(a, b, [-1.1], "fp64")
    V0 = torch.tensor(normal_block(p.n, 48, 3), device="cuda")
    run = lambda: f.slice_solve(0, -1.3, -0.9, V0, max_iter=3, check_every=3, allow_noconv=True)
    before = run()
    ctx.profile(["spmm_tc"])
    X = torch.tensor(normal_block(p.n, 64, 5), device="cuda")
    lam = torch.linspace(-3.0, -1.0, 64, dtype=torch.float64, device="cuda")
    ctx.selftest_alloc_limit(1 << 16)             # the lists of entries fail on the device, not those on the host
    ga, gb = sym.band_energy_grad(X, lam)
    ctx.selftest_alloc_limit()
    after = run()
    assert ctx.profile_query("spmm_tc")[0] > 0
    rows = torch.repeat_interleave(torch.arange(p.n, device="cuda"), torch.tensor(np.diff(p.rowptr), device="cuda"))
    cols = torch.tensor(p.colind, device="cuda").long()
    # 64 rounded products and sums of entries below 5
    assert torch.allclose(ga, (X[rows] * X[cols]).sum(1), rtol=0, atol=64 * 25 * 2e-16 * 64)
    assert torch.allclose(gb, -(X[rows] * lam * X[cols]).sum(1), rtol=0, atol=3 * 64 * 25 * 2e-16 * 64)
    # three iterations of the same start block: the same subspace up to rounding
    sel = before.resid < 1e-6
    assert sel.any() and np.abs(after.theta[sel] - before.theta[sel]).max() <= 1e-10


def test_lanczos_runs_hold_the_matrices_of_one_group(gpu_lib):
    # 64 runs of up to 256 steps on 64 rows: the vectors take 8.4 MB an array, the tridiagonal matrices of
    # all runs together would take 33.5 MB, those of 16 runs 8.4 MB
    p = laplacian_1d(64, mass=True)
    ctx, sym, a, b = setup(gpu_lib, p)
    x0 = normal_block(p.n, 64, 4)
    ctx.selftest_alloc_limit(12 << 20)
    runs = sym.dos_lanczos(a, b, 256, torch.tensor(x0, device="cuda"))
    A, B = p.dense("a"), p.dense("b")
    for c, (th, z2) in enumerate(runs):
        x = x0[:, c]
        quotient = (x @ A @ x) / (x @ B @ x)
        assert abs(z2.sum() - 1.0) <= 1e-10
        assert abs(z2 @ th - quotient) <= 1e-10 * np.abs(th).max()


def test_scratch_goes_back_on_request(gpu_lib):
    p = gaussian_pencil((9, 11, 11), (0.3, 2.0), seed=3)
    ctx, sym, a, b = setup(gpu_lib, p)
    X = torch.tensor(normal_block(p.n, 700, 5), device="cuda")
    lam = torch.linspace(-3.0, -1.0, 700, dtype=torch.float64, device="cuda")
    sym.band_energy_grad(X, lam)                  # lists of the pattern, modules
    ctx.release_scratch()
    free = torch.cuda.mem_get_info()[0]
    ga, _ = sym.band_energy_grad(X, lam)
    # 16 bytes an entry of X for each of two operands: 49 MB
    assert torch.cuda.mem_get_info()[0] <= free - 40e6
    ctx.release_scratch()
    assert torch.cuda.mem_get_info()[0] >= free - 4e6
    again, _ = sym.band_energy_grad(X, lam)
    assert torch.equal(ga, again)


def test_host_lists_that_do_not_fit(gpu_lib):
    # the lists of a pattern's tiles fail on the host: an out-of-memory status for the product, the CUDA cores
    # for the gradient, and both work once there is room
    p = gaussian_pencil((9, 11, 11), (0.3, 2.0), seed=3)
    ctx, sym, a, b = setup(gpu_lib, p)
    X = torch.tensor(normal_block(p.n, 64, 5), device="cuda")
    lam = torch.linspace(-3.0, -1.0, 64, dtype=torch.float64, device="cuda")
    ctx.selftest_alloc_limit(0)
    first, _ = sym.band_energy_grad(X, lam)
    with pytest.raises(gpu_lib.SisliceError, match="SS_ERR_OOM"):
        sym.spmm(a, b, X)
    ctx.selftest_alloc_limit()
    ctx.profile(["sddmm", "spmm_tc"])
    second, _ = sym.band_energy_grad(X, lam)
    Y = sym.spmm(a, b, X)
    ctx.profile_query("sddmm")
    assert ctx.profile_query_tensor("sddmm") > 0.0 and ctx.profile_query_tensor("spmm_tc") > 0.0
    xm = X.abs().max().item()
    assert (first - second).abs().max().item() <= 64 * 64 * 2.0 ** -52 * xm ** 2
    # n products of entries of A and X, cut 2^-53 below the largest
    ref = torch.tensor(p.dense("a"), device="cuda") @ X
    assert (Y - ref).abs().max().item() <= 8 * 2.0 ** -53 * p.n * float(np.abs(p.a).max()) * xm
