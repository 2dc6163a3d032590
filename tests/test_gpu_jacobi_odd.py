"""The one-block Jacobi eigensolver with an odd number of rotation pairs a round (Lanczos runs
of 49, 50 and 53 steps: 25 and 27 pairs), whose shared-memory arrays must stay aligned."""
import numpy as np
import pytest
import torch

from oracle import dos
from tests.gpu_util import setup
from workloads.pencils import gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [2, 49, 50, 53])
def test_odd_pair_counts(gpu_lib, steps):
    p = gaussian_pencil((4, 4, 4), seed=3)
    ctx, sym, a, b = setup(gpu_lib, p)
    X0 = normal_block(p.n, 2, 5)
    runs = sym.dos_lanczos(a, b, steps, torch.tensor(X0, device="cuda"))
    A, B = p.dense("a"), p.dense("b")
    for c in range(2):
        th_o, z_o, _, _ = dos.lanczos_ritz(A, B, X0[:, c], steps)
        th, z = runs[c]
        assert th.size == th_o.size
        assert np.abs(th - th_o).max() <= 1e-8 * np.abs(th_o).max()
        assert np.abs(z - z_o).max() <= 1e-8
