"""The two forms of the binary64 products (chfsi_set_fp64_products): exact digit
slices, the default, and FMAs on the ALUs, which also take over when the scratch
of the first does not fit.

Tolerances.  Blocks of random columns: 1e-13 for the cell products, 1e-12 for
overlap and rotation (as in test_gpu_digit_slices.py).  Entries spread over many
powers of two: the digit slices' bound K 2^-53 max|a| max|b| per sum of K terms,
once more for the reference's own rounding.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import ChfsiError, Context, workloads as W

from gpu_util import gpu_context, oracle_problem, rel_fro

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("p,ncol", [(1, 1), (2, 48), (4, 129), (6, 20), (8, 33)])
def test_alu_cell_products(p, ncol):
    s = W.small_periodic(seed=340 + p, ncell=3 if p <= 4 else 2, p=p, L=6.0, n_wells=4, n_want=10)
    ctx = gpu_context(s)
    try:
        X0 = W.start_block(s.seed, ctx.ndofs, ncol)
        X = torch.tensor(X0, device=DEV)
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        ref = oracle_problem(s).apply_Htilde(X0)
        ctx.set_fp64_operator("cells")
        ctx.apply(X, Z)
        ctx.set_fp64_products("alu")
        ctx.apply(X, Y)
        ctx.last_timings()
        assert rel_fro(Y.cpu().numpy(), ref) <= 1e-13
        assert not torch.equal(Y, Z)                  # the other kernels ran
    finally:
        ctx.destroy()


@pytest.mark.parametrize("mode", ["digits", "alu"])
@pytest.mark.parametrize("n", [1, 33, 129, 200])
def test_overlap_and_rotation(n, mode):
    ctx = Context(4, 8.0, 4)
    try:
        ctx.build()
        ctx.set_fp64_products(mode)
        ctx.set_blocking(90, 1)                       # X^T Y of two widths in the projection
        X0 = W.start_block(17 + n, ctx.ndofs, n)
        buf = torch.zeros((ctx.ndofs, n + 1), dtype=torch.float64, device=DEV)
        X = buf[:, :n]
        X.copy_(torch.tensor(X0))
        ctx.cholgs(X)
        ref = np.linalg.solve(np.linalg.cholesky(X0.T @ X0), X0.T).T
        assert rel_fro(X.cpu().numpy(), ref) <= 1e-12
        nfr = (n + 2) // 3                            # a narrow rotation, then a square one
        F = torch.empty((ctx.ndofs, nfr), dtype=torch.float64, device=DEV)
        dfr = ctx.rayleigh_ritz_split(X, F)
        d = ctx.rayleigh_ritz(X)
        scale = max(1.0, np.abs(d).max())
        assert np.abs(np.asarray(dfr) - d[n - nfr:]).max() <= 1e-12 * scale
        for V, ev in ((F, np.asarray(dfr)), (X, d)):
            Y = torch.empty(V.shape, dtype=torch.float64, device=DEV)
            ctx.apply(V, Y)
            h = (V.T @ Y).cpu().numpy()
            assert np.abs(h - np.diag(ev)).max() <= 1e-12 * scale
        assert bool((buf[:, n] == 0).all())
    finally:
        ctx.destroy()


def test_choice_is_checked():
    ctx = Context(2, 4.0, 2)
    try:
        with pytest.raises(ChfsiError):
            ctx._check(ctx._lib.chfsi_set_fp64_products(ctx._h, 2))
    finally:
        ctx.destroy()


def test_entries_far_apart_in_a_cell():
    """2^40 between the entries of a column: off by at most 8 cells of n_e terms of
    2^-53 max|H| max|X|, max|H| at most the spectral bound."""
    s = W.small_periodic(seed=350, ncell=3, p=4, L=6.0, n_wells=4, n_want=10)
    ctx = gpu_context(s)
    try:
        rng = np.random.default_rng(4)
        X0 = rng.uniform(-1.0, 1.0, (ctx.ndofs, 40)) * 2.0 ** -rng.uniform(0.0, 40.0, (ctx.ndofs, 40))
        X = torch.tensor(X0, device=DEV)
        Y = torch.empty_like(X)
        ctx.set_fp64_operator("cells")
        ctx.apply(X, Y)
        err = np.abs(Y.cpu().numpy() - oracle_problem(s).apply_Htilde(X0)).max()
        assert err <= 2 * 8 * 125 * 2.0 ** -53 * ctx.bounds(20) * np.abs(X0).max()
    finally:
        ctx.destroy()


def test_localised_columns():
    """Exponentially localised columns: the two forms differ in an entry by at most
    n 2^-53 of its row's largest times the rotation's largest of its column, each
    entry of the row relative to its column (and by what the factors differ)."""
    ctx = Context(4, 8.0, 4)
    try:
        ctx.build()
        n, M = 24, ctx.ndofs
        dist = np.abs(np.arange(M)[:, None] / M - np.arange(n)[None, :] / n)
        X0 = np.exp(-60.0 * dist) * (1.0 + 0.1 * W.start_block(5, M, n))
        out = {}
        for mode in ("digits", "alu"):
            ctx.set_fp64_products(mode)
            X = torch.tensor(X0, device=DEV)
            ctx.cholgs(X)
            out[mode] = X.cpu().numpy()
        Linv = np.linalg.inv(np.linalg.cholesky(X0.T @ X0))
        row = (np.abs(X0) / np.abs(X0).max(0)).max(1, keepdims=True)
        col = (np.abs(Linv) * np.abs(X0).max(0)).max(1)[None, :]
        # twice: the reference; and the factor, whose error is that of the overlap
        # times its condition number
        S = X0.T @ X0
        dinv = 1.0 / np.sqrt(np.diag(S))
        cond = np.linalg.cond(S * dinv[:, None] * dinv[None, :])
        bound = 2 * n * 2.0 ** -53 * row * col * (1.0 + n * cond)
        assert (np.abs(out["digits"] - out["alu"]) <= bound).all()
    finally:
        ctx.destroy()


@pytest.mark.parametrize("p,cells,ncol,op,alu", [
    (1, 14, 1, "default", True), (1, 14, 200, "default", True), (1, 5, 40, "default", False),
    (2, 17, 32, "cells", True), (2, 17, 33, "cells", False), (2, 10, 16, "cells", True), (2, 10, 17, "cells", False),
    (3, 17, 16, "cells", True), (3, 17, 17, "cells", False), (4, 12, 2, "cells", True), (4, 12, 3, "cells", False),
    (5, 9, 1, "cells", False), (7, 8, 1, "cells", True), (7, 8, 2, "cells", False),
    (4, 8, 12, "default", True), (4, 8, 13, "default", False)])
def test_widths_that_stay_on_the_alus(p, cells, ncol, op, alu):
    """Blocks for which the 128 x 48 tiles of the digit slices are a waste take the
    same kernels as with the products on the ALUs, and so the same bits."""
    ctx = Context(cells, 2.0 * cells, p)
    ctx.set_potential_gaussians([[1.0, 2.0, 3.0]], [2.0], [0.9])
    ctx.build()
    try:
        ctx.set_fp64_operator(op)
        g = torch.Generator(DEV).manual_seed(6)
        X = torch.randn((ctx.ndofs, ncol), device=DEV, generator=g, dtype=torch.float64)
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        ctx.apply(X, Y)
        ctx.set_fp64_products("alu")
        ctx.apply(X, Z)
        ctx.last_timings()
        assert torch.equal(Y, Z) == alu
        assert float((Y - Z).norm() / Z.norm()) <= 1e-13
    finally:
        ctx.destroy()
