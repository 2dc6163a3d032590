"""Lanczos runs asked for more steps than the pencil has rows: the Krylov space is full after N of them, what
is left of a vector is rounding, and the run ends there with weights that still sum to one."""
import numpy as np
import pytest
import torch

from tests.gpu_util import setup
from workloads.pencils import laplacian_1d, normal_block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [64, 65, 100, 256])
def test_runs_end_where_the_space_is_full(gpu_lib, steps):
    p = laplacian_1d(64, mass=True)
    ctx, sym, a, b = setup(gpu_lib, p)
    x0 = normal_block(p.n, 64, 4)
    runs = sym.dos_lanczos(a, b, steps, torch.tensor(x0, device="cuda"))
    A, B = p.dense("a"), p.dense("b")
    for c, (th, z2) in enumerate(runs):
        x = x0[:, c]
        quotient = (x @ A @ x) / (x @ B @ x)
        assert np.isfinite(th).all() and th.size <= steps
        assert abs(z2.sum() - 1.0) <= 1e-10
        assert abs(z2 @ th - quotient) <= 1e-10 * np.abs(th).max()
