"""Workloads of the library as its users run them, for timing and for comparing results.

Every case goes through the public Python entry points (``Context`` and
``Batch``), which call the C ABI of the same names.  The sizes are those of
the repository's workloads (the 4^3 cells, p = 4 system with 32 wanted states;
the 16^3 cells, p = 6 FCC supercell with 1,000; the p = 7 box with one
projector site per 4 bohr; the batch of uneven Dirichlet systems; the serving
requests of 2e4 to 2e6 unknowns) or lie between them.

``exact`` evaluates the same operations with plain torch in binary64 on the
global tensor-product grid (no cell loop): H~ = M^{-1/2} (1/2 K + V) M^{-1/2}
with 1-D mass, stiffness and Gauss-point matrices along each axis.
"""
import math

import numpy as np
import torch

from paper_1903_10959_gb300 import Batch, Context, fermi_level

DEV = "cuda"
DTYPE = {"fp64": torch.float64, "bf16x3": torch.float32, "mixed": torch.float32}


def listed():
    return [
        # one H~ X of the smallest system in binary64, as an iterative driver
        # around the library calls it: latency and launches count
        {"name": "apply_fp64_small", "kind": "apply", "nx": 4, "ny": 4, "nz": 4, "h": 2.5, "p": 4,
         "periodic": True, "n": 36, "prec": "fp64"},
        # a whole binary64 solve of that system: 10 iterations of degree 20 on
        # 32 states and 4 buffer states, then occupations and density
        {"name": "solve_fp64_small", "kind": "solve", "nx": 4, "ny": 4, "nz": 4, "h": 2.5, "p": 4,
         "periodic": True, "n": 36, "degree": 20, "iters": 10},
        # the filter of a serving request near the small end of its range
        {"name": "filter_request", "kind": "filter", "nx": 7, "ny": 7, "nz": 7, "h": 2.0, "p": 5,
         "periodic": True, "n": 77, "degree": 30, "prec": "bf16x3", "sites": 0},
        # the filter with separable projectors: p = 7, cells and sites as in
        # the 20^3-cell box of 1,000 sites
        {"name": "filter_projectors", "kind": "filter", "nx": 8, "ny": 8, "nz": 8, "h": 2.0, "p": 7,
         "periodic": True, "n": 330, "degree": 20, "prec": "bf16x3", "sites": 4},
        # the filter of the 16^3-cell FCC supercell with all 1,100 columns, the
        # largest part of a mixed-precision iteration
        {"name": "filter_large", "kind": "filter", "nx": 16, "ny": 16, "nz": 16, "h": 1.875, "p": 6,
         "periodic": True, "n": 1100, "degree": 40, "prec": "bf16x3", "sites": 0},
        # the same discretisation in binary64 on an eighth of the cells
        {"name": "filter_fp64", "kind": "filter", "nx": 8, "ny": 8, "nz": 8, "h": 1.875, "p": 6,
         "periodic": True, "n": 220, "degree": 40, "prec": "fp64", "sites": 0},
        # orthonormalisation of the full supercell block in mixed precision
        {"name": "cholgs_large", "kind": "cholgs", "nx": 16, "ny": 16, "nz": 16, "h": 1.875, "p": 6,
         "periodic": True, "n": 1100, "prec": "bf16x3"},
        # orthonormalisation in binary64
        {"name": "cholgs_fp64", "kind": "cholgs", "nx": 12, "ny": 12, "nz": 12, "h": 1.875, "p": 6,
         "periodic": True, "n": 550, "prec": "fp64"},
        # Rayleigh-Ritz in binary64, an odd number of states
        {"name": "rayleigh_ritz_fp64", "kind": "rr", "nx": 8, "ny": 8, "nz": 8, "h": 1.875, "p": 6,
         "periodic": True, "n": 333},
        # the batched filter over uneven isolated systems (a quarter of the
        # 64-system batch)
        {"name": "batch_filter", "kind": "batch", "count": 16, "p": 5, "h": 1.5, "degree": 30,
         "prec": "bf16x3"},
        # the next potential of an SCF-like sequence: new well depths, the cell
        # data rebuilt, and the first application on the warm block
        {"name": "rebuild_apply", "kind": "rebuild", "nx": 12, "ny": 12, "nz": 12, "h": 1.875, "p": 6,
         "periodic": True, "n": 110, "prec": "bf16x3"},
        # one application of the Bloch operator in mixed precision
        {"name": "kpoint_apply", "kind": "kpoint", "nx": 8, "ny": 8, "nz": 8, "h": 1.875, "p": 6,
         "periodic": True, "n": 110},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "solve", "filter", "filter", "projectors", "filter64", "cholgs", "cholgs",
                       "rr", "batch", "rebuild", "kpoint"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 16), "p": rng.choice([5, 5, 6]), "h": 1.5,
                "degree": rng.randint(10, 30), "prec": "bf16x3"}
    p = rng.randint(4, 7)

    def box(lo, hi):
        # unknowns over the range, the three sides uneven
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)) / 3.0) / p
        return {"n%s" % ax: max(2, int(round(side * rng.uniform(0.8, 1.2)))) for ax in "xyz"}

    per = rng.random() < 0.75
    h = round(rng.uniform(1.5, 2.5), 3)
    if kind == "apply":
        return {"kind": "apply", **box(3e3, 5e5), "h": h, "p": p, "periodic": per, "n": _log(rng, 1, 200),
                "prec": rng.choice(["fp64", "fp64", "bf16x3"])}
    if kind == "solve":
        return {"kind": "solve", **box(3e3, 2e4), "h": h, "p": p, "periodic": per, "n": _log(rng, 16, 64),
                "degree": rng.randint(15, 30), "iters": rng.randint(3, 10)}
    if kind == "filter":
        return {"kind": "filter", **box(1e4, 6e5), "h": h, "p": p, "periodic": per, "n": _log(rng, 20, 900),
                "degree": rng.randint(10, 40), "prec": rng.choice(["bf16x3", "bf16x3", "bf16x3", "mixed"]),
                "sites": 0}
    if kind == "projectors":
        return {"kind": "filter", **box(2e4, 2e5), "h": h, "p": rng.choice([6, 7]), "periodic": True,
                "n": _log(rng, 40, 330), "degree": rng.randint(10, 20), "prec": "bf16x3",
                "sites": rng.randint(2, 4)}
    if kind == "filter64":
        return {"kind": "filter", **box(5e3, 1.2e5), "h": h, "p": p, "periodic": per, "n": _log(rng, 16, 220),
                "degree": rng.randint(10, 40), "prec": "fp64", "sites": 0}
    if kind == "cholgs":
        prec = rng.choice(["bf16x3", "fp64"])
        return {"kind": "cholgs", **box(1e4, 8e5 if prec == "bf16x3" else 4e5), "h": h, "p": p, "periodic": per,
                "n": _log(rng, 16, 1100 if prec == "bf16x3" else 550), "prec": prec}
    if kind == "rr":
        return {"kind": "rr", **box(1e4, 1.2e5), "h": h, "p": p, "periodic": True, "n": _log(rng, 16, 333)}
    if kind == "rebuild":
        return {"kind": "rebuild", **box(1e4, 4e5), "h": h, "p": p, "periodic": per, "n": _log(rng, 20, 220),
                "prec": rng.choice(["bf16x3", "bf16x3", "fp64"])}
    return {"kind": "kpoint", **box(1e4, 1.2e5), "h": h, "p": p, "periodic": True, "n": _log(rng, 8, 220)}


# ---------------------------------------------------------------- problems
class _Problem:
    """Mesh and wells of one system, drawn from the seed."""

    def __init__(self, ncell, h, p, periodic, seed):
        self.ncell, self.p, self.periodic, self.seed = tuple(ncell), p, periodic, seed
        self.len = tuple(n * h for n in self.ncell)
        self.nd = tuple(n * p if periodic else n * p - 1 for n in self.ncell)
        self.m = self.nd[0] * self.nd[1] * self.nd[2]
        rng = np.random.default_rng([seed, 11])
        vol = self.len[0] * self.len[1] * self.len[2]
        nw = max(1, min(1000, int(round(vol / 105.0))))     # the supercell's density of wells
        lo, hi = (0.0, 1.0) if periodic else (0.1, 0.9)
        self.centres = (lo + (hi - lo) * rng.random((nw, 3))) * np.array(self.len)
        self.depths = 1.0 + 2.0 * rng.random(nw)
        self.widths = 0.8 + 0.4 * rng.random(nw)

    def context(self):
        c = Context(self.ncell, self.len, self.p, periodic=self.periodic)
        c.set_potential_gaussians(self.centres, self.depths, self.widths)
        return c

    def sites(self, per_side):
        """Projector sites on a jittered simple-cubic grid and their couplings."""
        rng = np.random.default_rng([self.seed, 12])
        g = (np.arange(per_side) + 0.5) / per_side
        xyz = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) * np.array(self.len)
        xyz = np.mod(xyz + 0.3 * rng.uniform(-1, 1, xyz.shape), np.array(self.len))
        return xyz, rng.uniform(0.5, 2.0, (len(xyz), 4))

    def window(self, n):
        """Filter bounds (a, b, a0): the top of the n wanted states, an upper bound
        of the spectrum and its lower end, from the free-particle estimate."""
        vol = self.len[0] * self.len[1] * self.len[2]
        ef = 0.5 * (6.0 * math.pi ** 2 * n / vol) ** (2.0 / 3.0)
        b = 12.0                                          # projectors, h <= 2 on |chi|^2 <= 6
        for d in range(3):
            x, w = _gll(self.p)
            B, D, gw = _basis(self.p)
            hh = self.len[d] / self.ncell[d]
            S = (D.T * gw) @ D * 2.0 / hh
            s = 1.0 / np.sqrt(w * hh / 2.0)
            b += 0.5 * float(np.linalg.eigvalsh(s[:, None] * S * s[None, :])[-1])
        return ef + 0.5, b, -2.5


def _problem(case, seed):
    return _Problem((case["nx"], case["ny"], case["nz"]), case["h"], case["p"], case["periodic"], seed)


def _block(pr, n, dtype, seed, grade=0.0, noise=0.05):
    """A block as a filter or a previous solve leaves it: M^{1/2}-weighted waves
    of the lowest n wavevectors, a few per cent of noise, columns graded from 1
    down to 10^-grade."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + 17)
    r = int(math.ceil((3.0 * n) ** (1.0 / 3.0))) + 2
    k = np.stack(np.meshgrid(*[np.arange(0, 2 * r)] * 3, indexing="ij"), -1).reshape(-1, 3)
    if pr.periodic:
        k = (k - r) * 2.0
    else:
        k = k + 1.0
    q = math.pi * k / np.array(pr.len)
    q = q[np.argsort((q * q).sum(1), kind="stable")[:n]]
    # of each pair k, -k one is the cosine and the other the sine
    first = np.where(q[:, 0] != 0, q[:, 0], np.where(q[:, 1] != 0, q[:, 1], q[:, 2]))
    phase = np.where(first < 0.0, 0.5 * math.pi, 0.0)
    mass = [torch.tensor(np.sqrt(m), device=DEV) for m in _mass_1d(pr)]
    X = torch.empty((pr.m, n), dtype=dtype, device=DEV)
    for c0 in range(0, n, 128):
        c1 = min(n, c0 + 128)
        w = []
        for d in range(3):
            x = torch.tensor(_nodes_1d(pr, d), device=DEV)
            t = x[:, None] * torch.tensor(q[c0:c1, d], device=DEV)[None, :]
            if pr.periodic:
                if d == 0:
                    t = t + torch.tensor(phase[c0:c1], device=DEV)[None, :]
                w.append(mass[d][:, None] * torch.polar(torch.ones_like(t), t))
            else:
                w.append((mass[d][:, None] * torch.sin(t)))
        yz = (w[2][:, None, :] * w[1][None, :, :]).reshape(-1, 1, c1 - c0).to(
            torch.complex64 if pr.periodic and dtype == torch.float32 else w[0].dtype)
        v = yz * w[0].to(yz.dtype)[None, :, :]
        v = (v.real if v.is_complex() else v).reshape(pr.m, c1 - c0).to(dtype)
        v *= 1.0 / v.norm(dim=0, keepdim=True)
        v += noise / math.sqrt(pr.m) * torch.randn(v.shape, dtype=dtype, device=DEV, generator=g)
        if grade:
            v *= torch.tensor(10.0 ** (-grade * np.arange(c0, c1) / max(1, n - 1)), dtype=dtype, device=DEV)
        X[:, c0:c1] = v
    return X


def _batch_problems(case, seed):
    """Uneven isolated systems: 4 to 12 cells a side, 16 to 400 states (at most M / 8)."""
    rng = np.random.default_rng([case["count"], 14])
    out = []
    for i in range(case["count"]):
        n = int(rng.integers(4, 13))
        m = (n * case["p"] - 1) ** 3
        nw = int(round(math.exp(rng.uniform(math.log(16), math.log(400)))))
        out.append((_Problem((n, n, n), case["h"], case["p"], False, 100 * seed + i),
                    max(8, min(int(nw * 1.1), m // 8))))
    return out


def _kvec(pr):
    return np.array([0.31, -0.17, 0.23]) * math.pi / np.array(pr.len)


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        prs = _batch_problems(case, seed)
        ctxs = []
        for pr, n in prs:
            c = pr.context()
            c.build()
            c.set_blocking(n, 1)
            ctxs.append(c)
        X0 = [_block(pr, n, torch.float32, 100 * seed + i, noise=0.2) for i, (pr, n) in enumerate(prs)]
        win = [pr.window(n) for pr, n in prs]
        return {"case": case, "batch": Batch(ctxs), "ctxs": ctxs, "X0": X0, "X": [torch.empty_like(x) for x in X0],
                "a": [w[0] for w in win], "b": [w[1] for w in win], "a0": [w[2] for w in win]}
    pr = _problem(case, seed)
    n = case["n"]
    ctx = pr.context()
    ctx.set_blocking(max(1, n), 1)
    s = {"case": case, "ctx": ctx, "pr": pr}
    if kind in ("apply", "rebuild"):
        s["X"] = _block(pr, n, DTYPE[case["prec"]], seed)
        s["Y"] = torch.empty_like(s["X"])
    if kind == "rebuild":
        s["next"] = _next_depths(pr, seed)
    if kind == "kpoint":
        s["X"] = torch.complex(_block(pr, n, torch.float32, seed), _block(pr, n, torch.float32, seed + 7919))
        s["Y"] = torch.empty_like(s["X"])
    if kind == "filter":
        if case["sites"]:
            ctx.set_projectors(*pr.sites(case["sites"]), sigma=0.8, rcut=3.0)
        s["window"] = pr.window(n)
        s["X0"] = _block(pr, n, DTYPE[case["prec"]], seed, noise=0.2)
        s["X"] = torch.empty_like(s["X0"])
    if kind == "cholgs":
        s["X0"] = _block(pr, n, DTYPE[case["prec"]], seed, grade=2.0)
        s["X"] = torch.empty_like(s["X0"])
    if kind == "rr":
        X = _block(pr, n, torch.float64, seed)
        s["X0"] = _orthonormal(X)
        s["X"] = torch.empty_like(X)
    if kind == "solve":
        s["X0"] = 2.0 * torch.rand((pr.m, n), dtype=torch.float64, device=DEV,
                                   generator=torch.Generator(device=DEV).manual_seed(seed + 5)) - 1.0
        s["X"] = torch.empty_like(s["X0"])
        s["b"] = pr.window(n)[1]
        s["rho"] = torch.empty(case["nx"] * case["ny"] * case["nz"] * (case["p"] + 2) ** 3, dtype=torch.float64,
                               device=DEV)
    ctx.build()
    if kind == "kpoint":
        ctx.set_kpoint(_kvec(pr))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        for x, x0 in zip(s["X"], s["X0"]):
            x.copy_(x0)
        s["batch"].filter(s["X"], case["degree"], s["a"], s["b"], s["a0"], prec=case["prec"])
        return s["X"]
    ctx = s["ctx"]
    if kind == "apply":
        ctx.apply(s["X"], s["Y"], prec=case["prec"])
        return s["Y"]
    if kind == "kpoint":
        ctx.apply_kpoint_mixed(s["X"], s["Y"])
        return s["Y"]
    if kind == "rebuild":
        ctx.set_potential_gaussians(s["pr"].centres, s["next"], s["pr"].widths)
        ctx.build()
        ctx.apply(s["X"], s["Y"], prec=case["prec"])
        return s["Y"]
    # the calls below work in place: each pass takes the block as it came
    X = s["X"]
    X.copy_(s["X0"])
    if kind == "filter":
        a, b, a0 = s["window"]
        ctx.filter(X, case["degree"], a, b, a0, prec=case["prec"])
        return X
    if kind == "cholgs":
        ctx.cholgs(X, prec=case["prec"])
        return X
    if kind == "rr":
        d = ctx.rayleigh_ritz(X)
        return {"evals": d, "X": X}
    # a whole solve; its eigenvectors are defined up to sign, so what a user's
    # next step takes from them, the density of all states, is the output
    d, _ = ctx.solve(X, case["iters"], case["degree"], s["b"])
    n = case["n"]
    _, occ = fermi_level(d, 0, float(n), 0.02)
    ctx.density(X, s["rho"], X, occ)
    return {"evals": d, "rho": s["rho"]}


# ---------------------------------------------------------------- the work
def _apply_flops(ncells, p):
    """Sum-factorised H_e of every cell on one vector."""
    n1, q = p + 1, p + 2
    return ncells * (14 * n1 ** 4 + 3 * n1 ** 3 + 4 * (q * n1 ** 3 + q * q * n1 ** 2 + q ** 3 * n1) + q ** 3)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        by = fl = 0
        for pr, n in _batch_problems(case, 0):
            by += 2 * pr.m * n * 4
            fl += case["degree"] * n * _apply_flops(pr.ncell[0] ** 3, case["p"])
        return {"bytes": by, "flops": fl}
    pr = _problem(case, 0)
    n, m = case["n"], pr.m
    cells = case["nx"] * case["ny"] * case["nz"]
    one = _apply_flops(cells, case["p"])
    es = 8 if case.get("prec", "fp64") == "fp64" else 4
    if kind == "apply":
        return {"bytes": 2 * m * n * es, "flops": n * one}
    if kind == "rebuild":
        n1, q = case["p"] + 1, case["p"] + 2
        form = 2 * cells * (q ** 3 * n1 ** 2 + q ** 2 * n1 ** 4 + q * n1 ** 6)
        return {"bytes": 2 * m * n * es, "flops": n * one + (form if es == 4 else 0)}
    if kind == "kpoint":
        return {"bytes": 2 * m * n * 8, "flops": 2 * n * one}
    if kind == "filter":
        return {"bytes": 2 * m * n * es, "flops": case["degree"] * n * one}
    if kind == "cholgs":
        return {"bytes": 2 * m * n * es, "flops": 2 * m * n * n + n ** 3}
    if kind == "rr":
        return {"bytes": 2 * m * n * 8, "flops": n * one + 3 * m * n * n + 9 * n ** 3}
    it = case["iters"]
    return {"bytes": 2 * m * n * 8,
            "flops": (it * (case["degree"] + 1) + 1) * n * one + (it + 1) * (5 * m * n * n + 10 * n ** 3)}


# ---------------------------------------------------------------- 64-bit values
def _legendre(n, x):
    """P_n and P_n' at x."""
    c = np.zeros(n + 1)
    c[n] = 1.0
    return (np.polynomial.legendre.legval(x, c),
            np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c)))


def _gll(p):
    c = np.zeros(p + 1)
    c[p] = 1.0
    d1 = np.polynomial.legendre.legder(c)
    d2 = np.polynomial.legendre.legder(d1)
    x = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.legroots(d1).real), [1.0]]) if p > 1 \
        else np.array([-1.0, 1.0])
    for _ in range(3):                                    # Newton on P_p'
        if p > 1:
            x[1:-1] -= np.polynomial.legendre.legval(x[1:-1], d1) / np.polynomial.legendre.legval(x[1:-1], d2)
    return x, 2.0 / (p * (p + 1) * _legendre(p, x)[0] ** 2)


def _basis(p):
    """Lagrange basis of the GLL nodes and its derivative at the p + 2 Gauss points, and their weights."""
    x, _ = _gll(p)
    g, gw = np.polynomial.legendre.leggauss(p + 2)
    B = np.ones((p + 2, p + 1))
    D = np.zeros((p + 2, p + 1))
    for i in range(p + 1):
        for j in range(p + 1):
            if j == i:
                continue
            D[:, i] = (D[:, i] * (g - x[j]) + B[:, i]) / (x[i] - x[j])
            B[:, i] = B[:, i] * (g - x[j]) / (x[i] - x[j])
    return B, D, gw


def _index_1d(pr, d):
    """Unknown index (or -1) of node i of cell c along axis d."""
    i = np.arange(pr.ncell[d])[:, None] * pr.p + np.arange(pr.p + 1)[None, :]
    if pr.periodic:
        return i % (pr.ncell[d] * pr.p)
    return np.where((i == 0) | (i == pr.ncell[d] * pr.p), -1, i - 1)


def _nodes_1d(pr, d):
    x, _ = _gll(pr.p)
    h = pr.len[d] / pr.ncell[d]
    out = np.zeros(pr.nd[d])
    idx = _index_1d(pr, d)
    pos = (np.arange(pr.ncell[d])[:, None] + 0.5 * (x[None, :] + 1.0)) * h
    out[idx[:, :-1][idx[:, :-1] >= 0]] = pos[:, :-1][idx[:, :-1] >= 0]
    return out


def _mass_1d(pr):
    _, w = _gll(pr.p)
    out = []
    for d in range(3):
        m = np.zeros(pr.nd[d] + 1)
        np.add.at(m, _index_1d(pr, d), np.broadcast_to(w * pr.len[d] / pr.ncell[d] / 2.0, (pr.ncell[d], pr.p + 1)))
        out.append(m[:-1])
    return out


class _Exact:
    """H~ of a problem on the whole grid, binary64."""

    def __init__(self, pr, depths=None, sites=0):
        self.pr = pr
        B, D, gw = _basis(pr.p)
        q = pr.p + 2
        self.A, self.S, self.C, self.B = [], [], [], []
        G = []
        gx = np.polynomial.legendre.leggauss(q)[0]
        self.xq, wq = [], []
        for d in range(3):
            h = pr.len[d] / pr.ncell[d]
            idx = _index_1d(pr, d)
            n = pr.nd[d]
            mats = [np.zeros((n + 1, n + 1)) for _ in range(3)]
            cell = [(B.T * gw) @ B * h / 2.0, (D.T * gw) @ D * 2.0 / h, (B.T * gw) @ D]
            for c in range(pr.ncell[d]):
                for m, e in zip(mats, cell):
                    np.add.at(m, np.ix_(idx[c], idx[c]), e)
            Bg = np.zeros((pr.ncell[d] * q, n + 1))
            for c in range(pr.ncell[d]):
                np.add.at(Bg, (np.arange(c * q, c * q + q)[:, None], idx[c][None, :]), B)
            s = np.concatenate([1.0 / np.sqrt(_mass_1d(pr)[d]), [0.0]])
            for lst, m in zip((self.A, self.S, self.C), mats):
                lst.append(torch.tensor((s[:, None] * m * s[None, :])[:n, :n], device=DEV))
            self.B.append(torch.tensor((Bg * s[None, :])[:, :n].copy(), device=DEV))
            x = ((np.arange(pr.ncell[d])[:, None] + 0.5 * (gx[None, :] + 1.0)) * h).reshape(-1)
            self.xq.append(x)
            wq.append(np.tile(gw * h / 2.0, pr.ncell[d]))
            im = (-1, 0, 1) if pr.periodic else (0,)
            G.append(sum(np.exp(-(x[None, :] - pr.centres[:, d:d + 1] - i * pr.len[d]) ** 2
                                / (2.0 * pr.widths[:, None] ** 2)) for i in im))
        dep = torch.tensor(pr.depths if depths is None else depths, device=DEV)
        g = [torch.tensor(x, device=DEV) for x in G]
        w = [torch.tensor(x, device=DEV) for x in wq]
        self.wq = w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]
        zy = (dep[:, None, None] * g[2][:, :, None] * g[1][:, None, :]).reshape(len(dep), -1)
        self.V = -(zy.T @ g[0]).reshape(self.wq.shape) * self.wq
        self.P = None
        if sites:
            self._projectors(*pr.sites(sites))

    def _projectors(self, xyz, h, sigma=0.8, rcut=3.0):
        rows = []
        for R in xyz:
            d = [torch.tensor(self.xq[a] - R[a], device=DEV) for a in range(3)]
            d = [v - L * torch.round(v / L) for v, L in zip(d, self.pr.len)]
            x, y, z = d[0][None, None, :], d[1][None, :, None], d[2][:, None, None]
            rr = x * x + y * y + z * z
            f = torch.where(rr <= rcut * rcut, torch.exp(-rr / (2.0 * sigma * sigma)), 0.0 * rr) * self.wq
            for t in (f, f * x / sigma, f * y / sigma, f * z / sigma):
                rows.append(self._back(t[..., None]).reshape(-1))
        self.P = torch.stack(rows)
        self.Ph = torch.tensor(h.reshape(-1), device=DEV)

    @staticmethod
    def _ax(m, u, axis):
        """Contract axis 0 (z), 1 (y) or 2 (x) of u (z, y, x, column) with m."""
        z, y, x, n = u.shape
        if axis == 0:
            return (m @ u.reshape(z, -1)).reshape(-1, y, x, n)
        if axis == 1:
            return torch.matmul(m, u.reshape(z, y, x * n)).reshape(z, -1, x, n)
        return torch.matmul(m, u.reshape(z * y, x, n)).reshape(z, y, -1, n)

    def _back(self, t):
        for axis, d in ((2, 0), (1, 1), (0, 2)):
            t = self._ax(self.B[d].T, t, axis)
        return t

    def cols(self, X, k=None):
        """H~ X (real), or with k the pair T = H~ + 1/2 |k|^2 A~ and k.G~ applied to X."""
        pr = self.pr
        u = X.reshape(pr.nd[2], pr.nd[1], pr.nd[0], -1)
        A, S, C = self.A, self.S, self.C
        az, sz = self._ax(A[2], u, 0), self._ax(S[2], u, 0)
        ayaz = self._ax(A[1], az, 1)
        out = 0.5 * (self._ax(S[0], ayaz, 2) + self._ax(A[0], self._ax(S[1], az, 1) + self._ax(A[1], sz, 1), 2))
        t = u
        for axis, d in ((0, 2), (1, 1), (2, 0)):
            t = self._ax(self.B[d], t, axis)
        out = out + self._back(t * self.V[..., None])
        if k is not None:
            out = out + 0.5 * float(k @ k) * self._ax(A[0], ayaz, 2)
            cz = self._ax(C[2], u, 0)
            kg = k[0] * self._ax(C[0], ayaz, 2) + self._ax(
                A[0], k[1] * self._ax(C[1], az, 1) + k[2] * self._ax(A[1], cz, 1), 2)
            return out.reshape(X.shape), kg.reshape(X.shape)
        out = out.reshape(X.shape)
        if self.P is not None:
            out = out + self.P.T @ (self.Ph[:, None] * (self.P @ X))
        return out

    def apply(self, X):
        step = max(1, int(4e8 // (8 * self.pr.m)))
        return torch.cat([self.cols(X[:, c:c + step].double()) for c in range(0, X.shape[1], step)], 1)

    def filter(self, X, degree, a, b, a0):
        e, c = (b - a) / 2.0, (b + a) / 2.0
        step = max(1, int(4e8 // (8 * self.pr.m)))
        out = []
        for c0 in range(0, X.shape[1], step):
            prev = X[:, c0:c0 + step].double()
            s1 = e / (a0 - c)
            sig = s1
            cur = (self.cols(prev) - c * prev) * (s1 / e)
            for _ in range(2, degree + 1):
                sn = 1.0 / (2.0 / s1 - sig)
                prev, cur = cur, (self.cols(cur) - c * cur) * (2.0 * sn / e) - sig * sn * prev
                sig = sn
            out.append(cur)
        return torch.cat(out, 1)


def _next_depths(pr, seed):
    """The well depths of the next step of a sequence: 1 % noise on the present ones."""
    rng = np.random.default_rng([seed, 15])
    return pr.depths * (1.0 + 0.01 * math.sqrt(3.0) * rng.uniform(-1.0, 1.0, pr.depths.shape))


def _orthonormal(X):
    X = X.double()
    for _ in range(2):
        L = torch.linalg.cholesky(X.T @ X)
        X = torch.linalg.solve_triangular(L, X.T, upper=False).T.contiguous()
    return X


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve" or work(case)["flops"] > 4e12 and kind in ("filter", "batch"):
        return None
    if kind == "batch":
        return [_Exact(pr).filter(_block(pr, n, torch.float32, 100 * seed + i, noise=0.2), case["degree"], *pr.window(n))
                for i, (pr, n) in enumerate(_batch_problems(case, seed))]
    pr = _problem(case, seed)
    n = case["n"]
    if kind == "kpoint":
        xr, xi = (_block(pr, n, torch.float32, t).double() for t in (seed, seed + 7919))
        op, k = _Exact(pr), _kvec(pr)
        step = max(1, int(4e8 // (8 * pr.m)))
        out = torch.empty((pr.m, n), dtype=torch.complex128, device=DEV)
        for c in range(0, n, step):
            (tr, gr), (ti, gi) = (op.cols(x[:, c:c + step], k) for x in (xr, xi))
            out[:, c:c + step] = torch.complex(tr + gi, ti - gr)
        return out
    if kind == "apply":
        return _Exact(pr).apply(_block(pr, n, DTYPE[case["prec"]], seed))
    if kind == "rebuild":
        return _Exact(pr, _next_depths(pr, seed)).apply(_block(pr, n, DTYPE[case["prec"]], seed))
    if kind == "filter":
        return _Exact(pr, sites=case["sites"]).filter(_block(pr, n, DTYPE[case["prec"]], seed, noise=0.2),
                                                      case["degree"], *pr.window(n))
    if kind == "cholgs":
        X = _block(pr, n, DTYPE[case["prec"]], seed, grade=2.0).double()
        L = torch.linalg.cholesky(X.T @ X)
        return torch.linalg.solve_triangular(L, X.T, upper=False).T
    X = _orthonormal(_block(pr, n, torch.float64, seed))
    h = X.T @ _Exact(pr).apply(X)
    # the rotated block is defined up to the sign of each column
    return {"evals": torch.linalg.eigvalsh(0.5 * (h + h.T)), "X": None}
