"""Cholesky factor and inverse of CholGS at the edges of its 32-column tiles,
against torch's binary64 factorisation of the same overlap matrix.

Tolerance: the columns are random with norms spread over 2^6, so the
column-scaled overlap has a condition number below 10 (n <= ndofs / 4); factor and
inverse each err by about n 2^-53 times it, 700 * 10 * 1.1e-16 = 8e-13 at the
largest n.  2e-12 on the orthonormal block, whose columns have norm one.
"""
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = Context(4, 8.0, 4)
    c.build()
    yield c
    c.destroy()


def block(ctx, n):
    X = torch.tensor(W.start_block(11 + n, ctx.ndofs, n), device=DEV)
    return X * 2.0 ** (torch.arange(n, device=DEV).double() % 7)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 250, 700])
def test_factor_and_inverse(ctx, n):
    X = block(ctx, n)
    Q = X.clone()
    ctx.cholgs(Q)
    L = torch.linalg.cholesky((X.T @ X).cpu())
    ref = torch.linalg.solve_triangular(L, X.T.cpu(), upper=False).T
    assert float((Q.cpu() - ref).norm(dim=0).max()) <= 2e-12


@pytest.mark.parametrize("n,bad", [(1, 0), (40, 0), (40, 31), (40, 32), (40, 39), (130, 77)])
def test_first_bad_pivot(ctx, n, bad):
    """A column of zeros: its pivot is reported and the block stays as it was."""
    X = block(ctx, n)
    X[:, bad:bad + 1] = 0.0
    Q = X.clone()
    with pytest.raises(RuntimeError, match="potrf info = %d$" % (bad + 1)):
        ctx.cholgs(Q)
    assert torch.equal(Q, X)
