"""Calls that only queue launches, recorded into a CUDA graph and replayed on new inputs: the band-energy
gradient at sizes that take the tensor cores outside a capture, a thin sparse product, and a solve with a
launch per level."""
import numpy as np
import pytest
import torch

from workloads.pencils import gaussian_pencil, normal_block

pytestmark = pytest.mark.gpu


def test_recorded_calls_match_direct_ones(gpu_lib):
    p = gaussian_pencil((9, 11, 11), (0.3, 2.0), seed=3)                   # N = 2,178
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gpu_lib.Context(0, stream)
        ctx.set_solve_mode("per_step")
        sym = ctx.analyze(p.rowptr, p.colind)
        a, b = torch.tensor(p.a, device="cuda"), torch.tensor(p.b, device="cuda")
        f = sym.factor(a, b, [-1.1], "fp64")
        lam = torch.linspace(-3.0, -1.0, 64, dtype=torch.float64, device="cuda")
        X = torch.tensor(normal_block(p.n, 64, 5), device="cuda")

        def calls():
            ga, gb = sym.band_energy_grad(X, lam)
            x = X[:, :4].contiguous()
            return ga, gb, sym.spmm(a, b, x), f.solve(0, x, refine=0)

        calls()
        ctx.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            recorded = calls()
        X.copy_(torch.tensor(normal_block(p.n, 64, 6), device="cuda"))
        graph.replay()
        stream.synchronize()
        got = [t.clone() for t in recorded]
        ref = calls()
        ctx.sync()
    xm = X.abs().max().item()
    # 64 products of entries below xm (lambda below 3); a sparse product's and a solve's rounding
    tols = (64 * 64 * 2.0 ** -52 * xm ** 2, 3 * 64 * 64 * 2.0 ** -52 * xm ** 2,
            p.n * 2.0 ** -52 * float(np.abs(p.a).max()) * xm,
            16 * p.n * 1.1e-16 * np.linalg.cond(p.dense("a") + 1.1 * p.dense("b")) * max(1.0, f.stats(0)[1])
            * ref[3].abs().max().item())
    for g, r, tol in zip(got, ref, tols):
        assert (g - r).abs().max().item() <= tol
