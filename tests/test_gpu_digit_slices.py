"""Binary64 products as exact digit slices on the tensor cores (cell products,
overlap and rotation) against plain binary64 of the same operation, at the
edges of the 128 x 48 output tiles, of the 16-deep chunks, of the segments of
192 terms and of the 960 terms between roundings.

Tolerances: the digit products are exact and each result is rounded once (and
once per 960 terms), so a product differs from the reference by the
reference's own rounding: at most K 2^-53 of sum |a||b|, in the norm about
sqrt(K) 2^-53 of it.  1e-13 covers the cell products (K <= 729, with the
amplification ||H~|| ||x|| / ||H~ x|| of up to a few hundred for smooth x; the
blocks here are random, amplification near 1); 1e-12 the overlap and rotation
(up to 1,000 columns, condition of the column-scaled blocks below 10).
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W

from gpu_util import gpu_context, oracle_problem, rel_fro

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("p,ncol", [(1, 1), (2, 48), (3, 37), (4, 1), (4, 129), (5, 47), (6, 128), (7, 13), (8, 20)])
@pytest.mark.parametrize("periodic", [True, False])
def test_cell_products(p, ncol, periodic):
    s = W.small_periodic(seed=300 + p, ncell=3 if p <= 5 else 2, p=p, L=6.0, n_wells=4, n_want=10)
    s.periodic = periodic
    prob = oracle_problem(s)
    ctx = gpu_context(s)
    try:
        # a view with an odd leading dimension and an odd column offset
        X0 = W.start_block(s.seed, prob.ndofs, ncol)
        buf = torch.zeros((prob.ndofs, ncol + 3), dtype=torch.float64, device=DEV)
        buf[:, 1:1 + ncol] = torch.tensor(X0, device=DEV)
        Y = torch.empty((prob.ndofs, ncol + 1), dtype=torch.float64, device=DEV)
        ctx.set_fp64_operator("cells")
        ctx.apply(buf[:, 1:1 + ncol], Y[:, :ncol])
        assert rel_fro(Y[:, :ncol].cpu().numpy(), prob.apply_Htilde(X0)) <= 1e-13
    finally:
        ctx.destroy()


@pytest.mark.parametrize("value", [1.0, float.fromhex("0x1.fffffffffffffp0"), -float.fromhex("0x1.fefefefefefefp0"),
                                   float.fromhex("0x1.01010101010102p-30")])
def test_extreme_digits(value):
    """Every entry the same: the digit sums add up instead of averaging out."""
    s = W.small_periodic(seed=310, ncell=4, p=6, L=8.0, n_wells=4, n_want=10)
    ctx = gpu_context(s)
    try:
        X = torch.full((ctx.ndofs, 50), value, dtype=torch.float64, device=DEV)
        X *= 2.0 ** (torch.arange(50, device=DEV).double() % 5)
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        ctx.apply(X, Y)
        ctx.set_fp64_operator("matrix-free")
        ctx.apply(X, Z)
        assert rel_fro(Y.cpu().numpy(), Z.cpu().numpy()) <= 1e-13
    finally:
        ctx.destroy()


@pytest.mark.parametrize("ncell,p,n", [(3, 2, 1), (3, 3, 16), (4, 4, 47), (4, 4, 48), (4, 4, 49), (3, 5, 97), (4, 4, 128),
                                       (4, 5, 129), (4, 6, 1000)])
def test_overlap_and_rotation(ncell, p, n):
    ctx = Context(ncell, 8.0, p)
    try:
        ctx.build()
        X0 = W.start_block(7 + n, ctx.ndofs, n)
        X0 *= 10.0 ** (-3.0 * np.arange(n) / max(1, n - 1))     # graded columns, as a filter leaves them
        buf = torch.zeros((ctx.ndofs, n + 1), dtype=torch.float64, device=DEV)
        X = buf[:, :n]
        X.copy_(torch.tensor(X0))
        ctx.cholgs(X)
        L = np.linalg.cholesky(X0.T @ X0)
        ref = np.linalg.solve(L, X0.T).T
        got = X.cpu().numpy()
        assert rel_fro(got, ref) <= 1e-12
        assert np.abs(got.T @ got - np.eye(n)).max() <= 1e-12
        # a full rotation: the Ritz values of the rotated block are its Rayleigh quotients
        d = ctx.rayleigh_ritz(X)
        Y = torch.empty_like(X)
        ctx.apply(X, Y)
        h = (X.T @ Y).cpu().numpy()
        assert np.abs(h - np.diag(d)).max() <= 1e-12 * max(1.0, np.abs(d).max())
    finally:
        ctx.destroy()


def test_not_finite():
    """An infinity or a NaN makes the values it enters NaN and no others."""
    s = W.small_periodic(seed=311, ncell=4, p=3, L=8.0, n_wells=2, n_want=10)
    ctx = gpu_context(s)
    try:
        X = torch.tensor(W.start_block(3, ctx.ndofs, 20), device=DEV)
        X[5, 3] = float("nan")
        X[77, 8] = float("inf")
        Y = torch.empty_like(X)
        ctx.set_fp64_operator("cells")
        ctx.apply(X, Y)
        bad = ~torch.isfinite(Y)
        assert bool(bad[:, 3].any()) and bool(bad[:, 8].any())
        bad[:, 3] = False
        bad[:, 8] = False
        assert not bool(bad.any())
    finally:
        ctx.destroy()
