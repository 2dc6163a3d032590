"""Refined solves of a shift that keeps its FP64 factor beside the FP32 one: few to many columns,
requested steps and a residual target, both products' modes; the residual is that of FP64."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["tensor", "simt"])
def test_refined_solves_reach_fp64(gpu_lib, mode):
    p = gaussian_pencil((10, 12, 11), seed=1)
    ctx, sym, a, b = setup(gpu_lib, p)
    ctx.set_gemm_mode(mode)
    f = sym.factor(a, b, [-1.1], "mixed")
    # usually FP64 + FP32 solves; the FP32 contraction that decides varies from run to run
    assert f.quality(0)[0] in ("mixed", "fp64+f32solve", "fp64")
    M = sp.csr_matrix((p.a + 1.1 * p.b, p.colind, p.rowptr), shape=(p.n, p.n))
    norm = abs(M).sum(axis=1).max()
    for k in (1, 7, 8, 9, 48):
        R = np.random.default_rng(k).standard_normal((p.n, k))
        for kw in ({"refine": 1}, {"refine": 2}):
            X = f.solve(0, torch.tensor(R, device="cuda"), **kw).cpu().numpy()
            # backward error n u of a refined solve
            res = np.linalg.norm(R - M @ X, axis=0)
            assert (res <= p.n * 1.1e-16 * (norm * np.linalg.norm(X, axis=0) + np.linalg.norm(R, axis=0))).all()
