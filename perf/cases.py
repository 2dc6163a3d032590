"""The library's work as a user's program has it done, case by case, through the public calls
of paper_1908_06043_gb300.api on seeded Gaussian-orbital pencils.

A case is a dict of plain values: the operation (``op``), the lattice of the pencil
(``lx`` x ``ly`` x ``lz`` atoms, ``fn`` functions each, N = lx ly lz fn rows) and the operation's
own sizes and options.  The sizes are those of the repository's benchmark and tests (N = 864 and
16,384; basis width 304; 1,640 eigenpairs; 8 to 16 windows; 4 Lanczos vectors of 100 steps; the
uneven batch of lattices of 8 to 18 atoms per axis with 2 or 4 functions).

What a program keeps between calls is kept here too: one context, and per lattice the pattern
and its symbolic analysis (made once per pattern, used for every shift and every pencil on it).
Everything else -- the atoms' potentials (and so A), right-hand sides, start blocks -- comes from
the seed; the kinetic and overlap parts of the pencil depend on the lattice alone, as in a
sequence of pencils on one basis.
"""
import math
from collections import OrderedDict

import numpy as np
import torch

from paper_1908_06043_gb300 import api

SPACING, DROP = 2.0, 1e-6
EXPONENTS = {2: (0.3, 2.0), 4: (0.3, 0.8, 2.0, 5.0)}
_CTX = []
_BASES = OrderedDict()


def _case(name, op, dims, fn, **kw):
    return dict(name=name, op=op, lx=dims[0], ly=dims[1], lz=dims[2], fn=fn, **kw)


def listed():
    big = (16, 16, 16)
    return [
        # one right-hand side on the smallest pencil: latency and launches
        _case("solve_one", "solve", (6, 6, 6), 4, sigma=-1.1, k=1, precision="fp64", refine=2),
        # a few right-hand sides, odd width, odd lattice
        _case("solve_thin", "solve", (15, 9, 17), 4, sigma=-0.9, k=7, precision="fp64", refine=1),
        # a probe's block solve where the rounded factor does not serve: FP64 throughout
        _case("solve_block_fp64", "solve", big, 4, sigma=-0.6, k=304, precision="fp64", refine=2),
        # a probe's block solve in the default precision: FP32 sweeps in FP64 refinement
        _case("solve_block_mixed", "solve", big, 4, sigma=-1.4, k=304, precision="mixed", refine=2),
        # one shift: factor, count the eigenvalues below it, solve with it
        _case("factor", "factor", big, 4, sigma=-1.3, k=1, precision="fp64", refine=2),
        # the window bounds of one pencil of the batch counted in one call
        _case("counts", "counts", (9, 12, 15), 2, shifts=9),
        # the residual product A X - B X diag(theta) of a probe
        _case("spmm_block", "spmm", big, 4, k=304, with_b=True),
        # the Lanczos sweep's product
        _case("spmm_thin", "spmm", big, 4, k=4, with_b=False),
        # the two products of one orthonormalisation step: Gram matrix, basis times factor
        _case("orthonormalise", "dense", big, 4, k=304),
        # the band-energy gradient over the wanted eigenvectors, sampled on the pattern
        _case("gradient", "gradient", big, 4, n_e=1640),
        # a whole window of a batch pencil: bounds counted, factored, solved, differentiated
        _case("window", "window", (10, 12, 11), 4, lo=-1.8, hi=-1.1, k=112, precision="fp64"),
        # the density-of-states estimate of a batch pencil
        _case("dos", "dos", (12, 8, 14), 2, steps=100, vectors=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, with sizes (odd ones among them) over the whole range."""
    op = rng.choice(["solve", "solve", "solve", "factor", "counts", "spmm", "dense", "gradient", "window", "dos"])
    fn = rng.choice([2, 4])
    top = {"window": 3500, "dos": 5000, "counts": 6000}.get(op, 16384)
    while True:
        dims = tuple(rng.randint(5, 18) for _ in range(3))
        if 600 <= dims[0] * dims[1] * dims[2] * fn <= top:
            break
    n = dims[0] * dims[1] * dims[2] * fn
    sigma = round(rng.uniform(-2.0, -0.4), 3)
    if op == "solve":
        return _case("", op, dims, fn, sigma=sigma, k=min(_log(rng, 1, 304), n // 2),
                     precision=rng.choice(["fp64", "mixed"]), refine=rng.choice([1, 2]))
    if op == "factor":
        return _case("", op, dims, fn, sigma=sigma, k=_log(rng, 1, 32), precision="fp64", refine=rng.choice([1, 2]))
    if op == "counts":
        return _case("", op, dims, fn, shifts=rng.randint(1, 9))
    if op == "spmm":
        return _case("", op, dims, fn, k=_log(rng, 1, 304), with_b=rng.random() < 0.5)
    if op == "dense":
        return _case("", op, dims, fn, k=_log(rng, 16, 304))
    if op == "gradient":
        return _case("", op, dims, fn, n_e=max(1, int(n * rng.uniform(0.01, 0.1))))
    if op == "window":
        lo = rng.uniform(-2.2, -1.2)
        return _case("", op, dims, fn, lo=round(lo, 3), hi=round(lo + 0.6, 3), k=16 * rng.randint(6, 9),
                     precision="fp64")
    return _case("", op, dims, fn, steps=4 * rng.randint(10, 25), vectors=rng.choice([1, 2, 4]))


# ------------------------------------------------------------------ the pencil of a case
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _context():
    if not _CTX:
        _CTX.append(api.Context(0 if torch.cuda.is_available() else -1))
    return _CTX[0]


class _Basis:
    """The part of a lattice's pencils that no potential changes: CSR pattern, kinetic and
    overlap values, the atoms of every entry, and the symbolic analysis."""

    def __init__(self, dims, fn):
        dev = _device()
        ex = torch.tensor(EXPONENTS[fn], dtype=torch.float64, device=dev)
        mu = ex[:, None] * ex[None, :] / (ex[:, None] + ex[None, :])
        pref = (2.0 * torch.sqrt(ex[:, None] * ex[None, :]) / (ex[:, None] + ex[None, :])) ** 1.5
        lx, ly, lz = dims
        atoms = lx * ly * lz
        i = torch.arange(atoms, device=dev)
        xyz = torch.stack([i % lx, (i // lx) % ly, i // (lx * ly)], dim=1)
        # no pair of functions of two atoms further apart than this reaches the drop limit
        reach2 = int((60.0 / float(mu.min())) / SPACING ** 2) + 1
        keys, ts, ss = [], [], []
        for a0 in range(0, atoms, 256):
            d = xyz[a0:a0 + 256, None, :] - xyz[None, :, :]
            r2s = (d * d).sum(dim=2)
            pi, pj = torch.nonzero(r2s <= reach2, as_tuple=True)
            r2 = r2s[pi, pj].to(torch.float64) * SPACING ** 2
            arg = mu * r2[:, None, None]
            s = pref * torch.exp(-arg)
            t = mu * (3.0 - 2.0 * arg) * s
            row = (pi + a0)[:, None, None] * fn + torch.arange(fn, device=dev)[None, :, None]
            col = pj[:, None, None] * fn + torch.arange(fn, device=dev)[None, None, :]
            keep = (s >= DROP) | (t.abs() >= DROP)
            keys.append((row * (atoms * fn) + col)[keep])
            ts.append(t[keep])
            ss.append(s[keep])
        key, order = torch.sort(torch.cat(keys))
        self.n = atoms * fn
        self.atoms, self.fn = atoms, fn
        self.t = torch.cat(ts)[order]
        self.b = torch.cat(ss)[order]
        self.row = key // self.n
        col = key % self.n
        self.row_atom, self.col_atom = self.row // fn, col // fn
        counts = torch.bincount(self.row, minlength=self.n)
        self.rowptr = np.zeros(self.n + 1, dtype=np.int64)
        np.cumsum(counts.cpu().numpy(), out=self.rowptr[1:])
        self.col = col
        self.colind = col.to(torch.int32).cpu().numpy()
        self.nnz = int(self.colind.size)
        self.sym = _context().analyze(self.rowptr, self.colind)

    def a(self, gen):
        v = -torch.rand(self.atoms, generator=gen, dtype=torch.float64, device=self.t.device)
        return self.t + 0.5 * (v[self.row_atom] + v[self.col_atom]) * self.b

    def dense(self, vals):
        m = torch.zeros(self.n * self.n, dtype=torch.float64, device=vals.device)
        m[self.row * self.n + self.col] = vals
        return m.view(self.n, self.n)

    def sparse(self, vals):
        return torch.sparse_csr_tensor(torch.tensor(self.rowptr, device=vals.device), self.col, vals,
                                       size=(self.n, self.n))


def _basis(case):
    key = (case["lx"], case["ly"], case["lz"], case["fn"])
    if key not in _BASES:
        while len(_BASES) >= 6:
            _BASES.popitem(last=False)
        _BASES[key] = _Basis(key[:3], key[3])
    _BASES.move_to_end(key)
    return _BASES[key]


# ------------------------------------------------------------------ inputs, one pass, exact values
def _inputs(case, seed):
    """What comes from the seed, and nothing of the library's."""
    bs = _basis(case)
    dev = bs.t.device
    gen = torch.Generator(device=dev).manual_seed(seed)
    s = dict(case=case, basis=bs, sym=bs.sym, a=bs.a(gen), b=bs.b)
    op, n = case["op"], bs.n

    def normal(k):
        return torch.randn(n, k, generator=gen, dtype=torch.float64, device=dev)

    if op in ("solve", "factor"):
        s["R"] = normal(case["k"])
    elif op == "counts":
        m = case["shifts"]
        s["sigmas"] = [-2.6 + 2.4 * (q + 0.5) / m for q in range(m)]
    elif op == "spmm":
        s["X"] = normal(case["k"])
        s["theta"] = None
        if case["with_b"]:
            u = torch.rand(case["k"], generator=gen, dtype=torch.float64, device=dev)
            s["theta"] = np.sort(-2.5 + 2.0 * u.cpu().numpy())
    elif op == "dense":
        k = case["k"]
        s["X"] = normal(k)
        s["Y"] = s["X"] + 0.1 * normal(k)
        s["Q"] = torch.tril(torch.randn(k, k, generator=gen, dtype=torch.float64, device=dev)) / math.sqrt(k)
    elif op == "gradient":
        s["X"] = normal(case["n_e"]) / math.sqrt(n)
        s["lam"] = torch.sort(-5.0 + 5.0 * torch.rand(case["n_e"], generator=gen, dtype=torch.float64,
                                                      device=dev))[0].contiguous()
    elif op == "window":
        s["V0"] = normal(case["k"])
    else:
        s["start"] = normal(case["vectors"])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["op"] == "solve":           # a program factors a shift once and solves with it many times
        s["factor"] = s["sym"].factor(s["a"], s["b"], [case["sigma"]], case["precision"])
    elif case["op"] == "dense":
        s["G"] = torch.empty(case["k"], case["k"], dtype=torch.float64, device=s["X"].device)
        s["Z"] = torch.empty_like(s["X"])
    return s


def _window(s):
    """The validated eigenpairs of one window, and their band energy with its gradient."""
    c, sym, kept = s["case"], s["sym"], {}

    def solver(a, b):
        f = sym.factor(a, b, [c["lo"], c["hi"]], "inertia")
        below = [f.inertia(0)[0], f.inertia(1)[0]]
        f.close()
        f = sym.factor(a, b, [0.5 * (c["lo"] + c["hi"])], c["precision"])
        pr = f.slice_solve(0, c["lo"], c["hi"], s["V0"], n_expect=max(1, below[1] - below[0]), check_every=3,
                           max_iter=80, allow_noconv=True)
        f.close()
        sel = np.nonzero((pr.theta > c["lo"]) & (pr.theta <= c["hi"]) & (pr.resid <= 1e-10))[0]
        kept["below"], kept["theta"] = np.array(below), np.zeros(c["k"])
        kept["theta"][:sel.size] = pr.theta[sel]
        dev = pr.X.device
        return torch.tensor(pr.theta[sel], device=dev), pr.X[:, torch.as_tensor(sel, device=dev)].contiguous()

    a = s["a"].detach().requires_grad_(True)
    b = s["b"].detach().requires_grad_(True)
    e = api.BandEnergy.apply(a, b, sym, solver)
    e.backward()
    return {"below": kept["below"], "theta": kept["theta"], "energy": e.detach(), "grad_a": a.grad, "grad_b": b.grad}


def run(s):
    c, sym = s["case"], s["sym"]
    op = c["op"]
    if op == "solve":
        return s["factor"].solve(0, s["R"], refine=c["refine"])
    if op == "factor":
        f = sym.factor(s["a"], s["b"], [c["sigma"]], c["precision"])
        neg, zero, pos, _ = f.inertia(0)
        x = f.solve(0, s["R"], refine=c["refine"])
        f.close()
        return {"inertia": np.array([neg, zero, pos]), "x": x}
    if op == "counts":
        f = sym.factor(s["a"], s["b"], s["sigmas"], "inertia")
        got = np.array([f.inertia(j)[0] for j in range(len(s["sigmas"]))])
        f.close()
        return got
    if op == "spmm":
        if s["theta"] is None:
            return sym.spmm(s["a"], s["b"], s["X"])
        return sym.spmm(s["a"], s["b"], s["X"], 1.0, -s["theta"])
    if op == "dense":
        g = sym.ctx.dense_gram(s["X"], s["Y"], s["G"])
        z = sym.ctx.dense_gemm(s["X"], s["Q"], s["Z"], transq=True)
        return {"gram": g, "basis": z}
    if op == "gradient":
        ga, gb = sym.band_energy_grad(s["X"], s["lam"])
        return {"grad_a": ga, "grad_b": gb}
    if op == "window":
        return _window(s)
    runs = sym.dos_estimate(s["a"], s["b"], c["steps"], s["start"])
    return {"theta": np.stack([r[0] for r in runs]), "weight": np.stack([r[1] for r in runs])}


def exact(case, seed):
    """What run() returns, from plain torch in 64 bits (dense where the operation needs an inverse)."""
    op = case["op"]
    if op == "window" or op == "dos":
        return None
    s = _inputs(case, seed)
    bs, a, b = s["basis"], s["a"], s["b"]
    if op == "solve" or op == "factor":
        m = bs.dense(a - case["sigma"] * b)
        x = torch.linalg.solve(m, s["R"])
        x += torch.linalg.solve(m, s["R"] - m @ x)
        return x if op == "solve" else {"inertia": None, "x": x}
    if op == "counts":
        return None
    if op == "spmm":
        y = bs.sparse(a) @ s["X"]
        if s["theta"] is not None:
            y -= (bs.sparse(b) @ s["X"]) * torch.tensor(s["theta"], device=y.device)
        return y
    if op == "dense":
        return {"gram": s["X"].T @ s["Y"], "basis": s["X"] @ s["Q"].T}
    x, lam = s["X"], s["lam"]
    ga, gb = (x @ x.T).view(-1), ((x * lam) @ x.T).view(-1)
    at = bs.row * bs.n + bs.col
    return {"grad_a": ga[at], "grad_b": -gb[at]}


def work(case):
    """Bytes (each input read once, each output written once) and algorithmic flops of one pass."""
    bs, op = _basis(case), case["op"]
    n, nnz, info = bs.n, bs.nnz, bs.sym.info
    vals, ell = 16.0 * nnz + 4.0 * nnz, 8.0 * (info["l_offdiag_entries"] + info["l_diag_entries"])
    sweep = 4.0 * info["l_offdiag_entries"] + 2.0 * info["l_diag_entries"]
    if op == "solve":
        k, r = case["k"], case["refine"]
        return {"bytes": ell + (vals if r else 0) + 16.0 * n * k, "flops": k * (sweep * (r + 1) + 2.0 * nnz * r)}
    if op == "factor":
        k, r = case["k"], case["refine"]
        return {"bytes": vals + ell + 16.0 * n * k, "flops": info["factor_flops"] + k * (sweep * (r + 1) + 2.0 * nnz * r)}
    if op == "counts":
        return {"bytes": vals, "flops": info["factor_flops"] * case["shifts"]}
    if op == "spmm":
        m = 2 if case["with_b"] else 1
        return {"bytes": (8.0 * m + 4.0) * nnz + 16.0 * n * case["k"], "flops": 2.0 * m * nnz * case["k"]}
    if op == "dense":
        k = case["k"]
        return {"bytes": 8.0 * (3.0 * n * k + 2.0 * k * k), "flops": 3.0 * n * k * k}
    if op == "gradient":
        return {"bytes": 8.0 * n * case["n_e"] + 20.0 * nnz, "flops": 4.0 * nnz * case["n_e"]}
    if op == "window":
        # three factorisations and, at the least, one solve and two products a column of the window's basis
        k = case["k"]
        return {"bytes": vals + ell + 16.0 * n * k, "flops": 3.0 * info["factor_flops"] + k * (sweep + 4.0 * nnz)}
    m, k = case["steps"], case["vectors"]
    return {"bytes": vals + ell + 8.0 * n * k, "flops": info["factor_flops"] + m * k * (sweep + 4.0 * nnz + 4.0 * m * n)}
