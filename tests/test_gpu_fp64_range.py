"""Binary64 products at the ends of the exponent range: columns so small or large
that products of their entries, or the entries themselves, are subnormal numbers
or close to overflow.

Tolerances.  A result that is rounded to a multiple of 2^-1074 is off by half of
that; the overlap of M rows adds up to 32 such sums, the application 8 per cell
row of 125 products (the ALU form rounds each product).  Else 1e-12 for the
orthonormalised block and 1e-13 for the application, as in the other tests.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N = 40


@pytest.fixture(scope="module")
def system():
    ctx = Context(4, 8.0, 4)
    ctx.build()
    X = torch.tensor(W.start_block(3, ctx.ndofs, N), device=DEV)
    yield ctx, X
    ctx.destroy()


@pytest.mark.parametrize("mode", ["digits", "alu"])
@pytest.mark.parametrize("k", [-530, -520, -515, -510, -505, -400, 0, 400, 500, 504])
def test_cholgs(system, k, mode):
    """Columns of size 2^k: the overlap's entries are of size 2^(2k)."""
    ctx, X0 = system
    ctx.set_fp64_products(mode)
    try:
        X = X0 * 2.0 ** k
        ctx.cholgs(X)
    finally:
        ctx.set_fp64_products("digits")
    # off-diagonal errors of the overlap relative to its diagonal, n of them per
    # entry of the product with the inverse factor (condition below 2)
    smallest = float((X0 * X0).sum(0).min())
    step = 2.0 ** (-1074 - 2 * k) / smallest if k < -400 else 0.0
    err = float((X.T @ X - torch.eye(N, dtype=torch.float64, device=DEV)).abs().max())
    assert err <= 1e-12 + (32 if mode == "digits" else ctx.ndofs) * 2 * N * step


@pytest.mark.parametrize("mode", ["digits", "alu"])
@pytest.mark.parametrize("k", [-1073, -1060, -1040, -1020, -1000, 0, 1000, 1010])
def test_application(system, k, mode):
    ctx, X0 = system
    ref = torch.empty_like(X0)
    ctx.apply(X0, ref)
    ctx.set_fp64_operator("cells")
    ctx.set_fp64_products(mode)
    try:
        X = torch.tensor(np.ldexp(X0.cpu().numpy(), k), device=DEV)
        Y = torch.empty_like(X)
        ctx.apply(X, Y)
        if k < -1000:                                   # the entries as they were rounded
            exact = torch.tensor(np.ldexp(X.cpu().numpy(), -k), device=DEV)
            ctx.apply(exact, ref)
        ctx.last_timings()
    finally:
        ctx.set_fp64_products("digits")
        ctx.set_fp64_operator("default")
    got, want = Y.cpu().numpy(), ref.cpu().numpy()
    err = np.abs(np.ldexp(np.ldexp(got, -k // 2), -k - (-k // 2)) - want).max()
    assert err <= 1e-13 * np.abs(want).max() + 8 * 125 * 2.0 ** min(0, max(-1074 - k, -200))
    assert bool((Y != 0).any()) or k < -1070


def test_column_of_subnormal_numbers_beside_normal_ones(system):
    """Each column has its own scale."""
    ctx, X0 = system
    X = X0.clone()
    X[:, 7] = torch.tensor(np.ldexp(X0[:, 7].cpu().numpy(), -1050), device=DEV)
    Y, ref = torch.empty_like(X), torch.empty_like(X)
    ctx.set_fp64_operator("cells")
    ctx.apply(X, Y)
    ctx.apply(X0, ref)
    ctx.set_fp64_operator("default")
    ctx.last_timings()
    keep = [c for c in range(N) if c != 7]
    assert torch.equal(Y[:, keep], ref[:, keep])
    assert bool((Y[:, 7] != 0).any())
