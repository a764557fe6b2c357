"""Binary64 digit-slice products in several launches each: the words of a launch
take 512 MB at most, so 132,651 rows of 701 columns are cut into two slices of
the overlap and of the rotation and three of the cells, the last one shorter.

Tolerances as for the single-launch products: 1e-13 for the cell products
against the sum-factorised operator, 1e-12 for the overlap and the rotation
(condition of the random block below 2).
"""
import pytest
import torch

from paper_1903_10959_gb300 import Context

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def system():
    ctx = Context(13, 26.0, 4, periodic=False)
    ctx.set_potential_gaussians([[7.0, 12.0, 19.0], [15.0, 3.0, 9.0]], [2.0, 3.0], [1.0, 0.8])
    ctx.build()
    g = torch.Generator(device=DEV)
    g.manual_seed(5)
    X = 2.0 * torch.rand((ctx.ndofs, 701), dtype=torch.float64, device=DEV, generator=g) - 1.0
    ctx.set_blocking(701, 1)
    yield ctx, X
    ctx.destroy()


def test_cell_products(system):
    ctx, X = system
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    ctx.set_fp64_operator("cells")
    ctx.apply(X, Y)
    ctx.set_fp64_operator("matrix-free")
    ctx.apply(X, Z)
    ctx.set_fp64_operator("default")
    ctx.last_timings()
    err = (Y - Z).norm(dim=0) / Z.norm(dim=0)
    assert float(err.max()) <= 1e-13


def test_overlap_and_rotation(system):
    ctx, X = system
    Q = X.clone()
    ctx.cholgs(Q)
    L = torch.linalg.cholesky(X.T @ X)
    ref = torch.linalg.solve_triangular(L, X.T, upper=False).T
    assert float((Q - ref).norm() / ref.norm()) <= 1e-12
    assert float((Q.T @ Q - torch.eye(701, dtype=torch.float64, device=DEV)).abs().max()) <= 1e-12


def test_projection_of_a_narrower_block(system):
    """X^T Y of two blocks (Rayleigh-Ritz in column blocks of 200)."""
    ctx, X = system
    Q = X.clone()
    ctx.cholgs(Q)
    ctx.set_blocking(200, 1)
    d = ctx.rayleigh_ritz(Q)
    ctx.set_blocking(701, 1)
    Y = torch.empty_like(Q)
    ctx.apply(Q, Y)
    h = Q.T @ Y
    assert float((h - torch.diag(torch.tensor(d, device=DEV))).abs().max()) <= 1e-12 * float(abs(d).max())
