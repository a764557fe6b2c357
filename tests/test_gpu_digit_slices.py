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
