"""Refined solves of a shift that has both an FP64 factor and its FP32 rounding (precision "mixed_tc" keeps both
wherever the rounded copy contracts): requested steps, and the residual target of a probe's solves, run in FP64,
shown by the kernels that are timed."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu

SIGMA = -6.0          # below the spectrum: the rounded copy of a definite matrix contracts


def factored(gpu_lib, mode):
    p = gaussian_pencil((6, 8, 9), seed=5)                                # N = 1,728
    ctx, sym, a, b = setup(gpu_lib, p)
    ctx.set_gemm_mode(mode)
    f = sym.factor(a, b, [SIGMA], "mixed_tc")
    assert f.quality(0)[0] == "fp64+f32solve"
    return p, ctx, f


@pytest.mark.parametrize("mode", ["tensor", "simt"])
@pytest.mark.parametrize("k", [1, 7, 8, 9, 48, 128])
def test_requested_steps(gpu_lib, mode, k):
    p, ctx, f = factored(gpu_lib, mode)
    M = sp.csr_matrix((p.a - SIGMA * p.b, p.colind, p.rowptr), shape=(p.n, p.n))
    norm = abs(M).sum(axis=1).max()
    R = np.random.default_rng(k).standard_normal((p.n, k))
    for steps in (1, 2):
        ctx.profile(["solve", "solve_f32"])
        X = f.solve(0, torch.tensor(R, device="cuda"), refine=steps).cpu().numpy()
        count, count32 = ctx.profile_query("solve")[0], ctx.profile_query("solve_f32")[0]
        ctx.profile()
        # 895,300 entries of L on 21 levels: FP64 up to 469 columns on either path
        assert (count, count32) == (steps + 1, 0)
        # backward error n u of a refined solve
        res = np.linalg.norm(R - M @ X, axis=0)
        assert (res <= p.n * 1.1e-16 * (norm * np.linalg.norm(X, axis=0) + np.linalg.norm(R, axis=0))).all()


@pytest.mark.parametrize("mode", ["tensor", "simt"])
@pytest.mark.parametrize("k", [8, 96])
def test_residual_target_of_a_probe(gpu_lib, mode, k):
    p, ctx, f = factored(gpu_lib, mode)
    V0 = torch.tensor(normal_block(p.n, k, 3), device="cuda")
    ctx.profile(["solve", "solve_f32"])
    r = f.slice_solve(0, SIGMA, 0.0, V0, max_iter=4, check_every=4, refine_from_start=True, allow_noconv=True)
    count, count32 = ctx.profile_query("solve")[0], ctx.profile_query("solve_f32")[0]
    ctx.profile()
    # every solve ends at the target, 1e-13 of the right-hand side, or after 12 corrections
    assert r.iterations == 4 and count32 == 0
    assert count == r.iterations + r.refine_steps and r.refine_steps <= 12 * r.iterations
    # the returned values are Rayleigh quotients of the returned vectors
    X = r.X.cpu().numpy()
    A, B = (sp.csr_matrix((v, p.colind, p.rowptr), shape=(p.n, p.n)) for v in (p.a, p.b))
    quotient = (X * (A @ X)).sum(0) / (X * (B @ X)).sum(0)
    assert np.abs(r.theta - quotient).max() <= 1e-9 * np.abs(quotient).max()
    # four inverse iterations of a definite operator bring the lowest pair below 1e-3 from a random start
    assert r.resid.min() <= 1e-3
