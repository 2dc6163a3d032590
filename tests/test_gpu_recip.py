"""The reciprocal of the diagonal blocks' pivots against the division: random mantissas, those next to powers
of two, both signs, every exponent, and the exponents around 2^+-1000 where the division takes over."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def bits(x):
    return np.ascontiguousarray(x).view(np.int64)


def test_reciprocals_within_one_unit(gpu_lib):
    rng = np.random.default_rng(1)
    m = 1 << 20
    mant = rng.integers(0, 1 << 52, m)
    edge = np.concatenate([np.arange(512), (1 << 52) - 1 - np.arange(512)])
    mant[:edge.size] = edge
    exps = np.concatenate([rng.integers(1, 2047, m // 2), rng.integers(20, 27, m // 8), rng.integers(2020, 2027, m // 8),
                           rng.integers(1020, 1027, m // 4)])
    rng.shuffle(exps)
    d = ((rng.integers(0, 2, m) << 63) | (exps << 52) | mant).astype(np.int64).view(np.float64)
    ctx = gpu_lib.Context(0)
    got = ctx.selftest_recip(torch.tensor(d, device="cuda")).cpu().numpy()
    ref = 1.0 / d
    assert np.abs(bits(got) - bits(ref)).max() <= 1
    far = (exps < 23) | (exps > 2023)
    assert far.any() and (got[far] == ref[far]).all()


def test_special_values(gpu_lib):
    d = np.array([0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324, 2.0 ** -1000, 2.0 ** 1000, 1.0, -1.0, np.nan])
    got = gpu_lib.Context(0).selftest_recip(torch.tensor(d, device="cuda")).cpu().numpy()
    ref = np.array([0.0, 0.0, 0.0, -0.0, np.inf, -np.inf, 2.0 ** 1000, 2.0 ** -1000, 1.0, -1.0])
    assert (got[:10] == ref).all() and np.isnan(got[10])
