"""Cholesky factor and inverse of CholGS where a step has more tiles than groups of
warps (605 on 152 SMs, from 35 block columns on), and an overlap that is not finite.

Tolerance: as for the small sizes, n 2^-53 times the condition number of the
column-scaled overlap (below 10) for the factor and again for the inverse: 3.4e-12
at n = 1,505.
"""
import pytest
import torch

from paper_1903_10959_gb300 import ChfsiError, Context

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = Context(8, 16.0, 3)
    c.build()
    yield c
    c.destroy()


def block(ctx, n):
    g = torch.Generator(DEV).manual_seed(21 + n)
    X = 2.0 * torch.rand((ctx.ndofs, n), dtype=torch.float64, device=DEV, generator=g) - 1.0
    return X * 2.0 ** (torch.arange(n, device=DEV).double() % 7)


@pytest.mark.parametrize("n", [1089, 1100, 1505])
def test_factor_and_inverse(ctx, n):
    X = block(ctx, n)
    Q = X.clone()
    ctx.cholgs(Q)
    L = torch.linalg.cholesky(X.T @ X)
    ref = torch.linalg.solve_triangular(L, X.T, upper=False).T
    assert float((Q - ref).norm(dim=0).max()) <= 3.4e-12


@pytest.mark.parametrize("mode", ["digits", "alu"])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n,bad", [(1, 0), (40, 39), (130, 5), (130, 64)])
def test_overlap_that_is_not_finite(ctx, n, bad, value, mode):
    """A NaN or an infinity in one column: its pivot is reported, no other entry of
    the overlap is touched, and the block stays as it was."""
    X = block(ctx, n)
    X[777, bad] = value
    Q = X.clone()
    ctx.set_fp64_products(mode)
    try:
        with pytest.raises(ChfsiError, match="potrf info = %d$" % (bad + 1)) as e:
            ctx.cholgs(Q)
    finally:
        ctx.set_fp64_products("digits")
    assert e.value.status == 4                        # CHFSI_ERR_NOT_SPD
    assert torch.equal(Q.nan_to_num(3.5), X.nan_to_num(3.5))
