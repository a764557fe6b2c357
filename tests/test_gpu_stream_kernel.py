"""The BF16x3 cell kernel of one thread block per SM against the ring kernel: the
same bits for every number of nodes, row parts and chunks per cell, Dirichlet
rows, ragged tiles and unaligned blocks, with projector and Bloch chunks and in
the FP16x2 form.

Launches of 304 items (cell, 128-column tile, row part) and more take it on 152
SMs, so the reference comes from another kernel or from column blocks below that.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import ChfsiError, Context

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _ctx(p, n, periodic=True, sites=0):
    rng = np.random.default_rng(p)
    L = 2.0 * n
    ctx = Context(n, L, p, periodic=periodic)
    ctx.set_potential_gaussians(L * rng.random((5, 3)), 1.0 + rng.random(5), 0.6 + rng.random(5))
    if sites:
        ctx.set_projectors(L * rng.random((sites, 3)), rng.uniform(0.3, 1.0, (sites, 4)), sigma=0.8, rcut=3.0)
    ctx.build()
    return ctx


def _block(ctx, n, seed=3, dtype=torch.float32):
    g = torch.Generator(DEV).manual_seed(seed)
    return torch.randn((ctx.ndofs, n), device=DEV, generator=g, dtype=dtype)


@pytest.mark.parametrize("p,cells", [(1, 13), (2, 9), (3, 7), (4, 6), (5, 7), (6, 6), (7, 5), (8, 5)])
@pytest.mark.parametrize("ncol,ld,off", [(129, 132, 0), (256, 256, 0), (131, 133, 1), (40, 40, 0)])
def test_same_bits_as_the_rings(p, cells, ncol, ld, off):
    ctx = _ctx(p, cells, periodic=ncol != 129)
    try:
        X = _block(ctx, ld)[:, off:off + ncol]
        Y, Z = (torch.full((ctx.ndofs, ld), float("nan"), device=DEV)[:, off:off + ncol] for _ in range(2))
        ctx.set_cell_gather("rings4")
        ctx.apply(X, Z, prec="bf16x3")
        ctx.set_cell_gather("rings")
        ctx.apply(X, Y, prec="bf16x3")
        assert torch.equal(Y, Z)
    finally:
        ctx.destroy()


@pytest.mark.parametrize("p,cells,sites,prec", [(2, 6, 4, "bf16x3"), (5, 5, 3, "bf16x3"), (6, 5, 80, "bf16x3"),
                                               (7, 4, 20, "bf16x3"), (3, 6, 0, "f16x2"), (5, 5, 0, "f16x2"),
                                               (6, 5, 0, "f16x2"), (8, 4, 0, "f16x2")])
def test_against_narrow_blocks(p, cells, sites, prec):
    ctx = _ctx(p, cells, sites=sites)
    try:
        X = _block(ctx, 400)
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        ctx.apply(X, Y, prec=prec)
        for c in range(0, 400, 40):                        # one tile: the ring kernel
            x, z = X[:, c:c + 40].contiguous(), torch.empty((ctx.ndofs, 40), device=DEV)
            ctx.apply(x, z, prec=prec)
            Z[:, c:c + 40] = z
        assert torch.equal(Y, Z)
    finally:
        ctx.destroy()


@pytest.mark.parametrize("p,cells", [(3, 6), (5, 4), (6, 4)])
def test_bloch_chunks(p, cells):
    ctx = _ctx(p, cells)
    try:
        ctx.set_kpoint([0.31, -0.17, 0.44])
        X = _block(ctx, 400).view(ctx.ndofs, 200, 2)
        X = torch.view_as_complex(X.contiguous())
        Y = torch.empty_like(X)
        ctx.apply_kpoint_mixed(X, Y)
        for c in range(0, 200, 50):
            x = X[:, c:c + 50].contiguous()
            z = torch.empty_like(x)
            ctx.apply_kpoint_mixed(x, z)
            assert torch.equal(Y[:, c:c + 50], z)
    finally:
        ctx.destroy()


def test_bounded_waits():
    """A withheld arrival runs the waits of one block out: an error, and the context
    goes on (ERR_TIMEOUT; the hook is off by default)."""
    ctx = _ctx(5, 7)
    try:
        X = _block(ctx, 40)
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        ctx.apply(X, Y, prec="bf16x3")
        ctx.debug_withhold_arrival(True)
        try:
            with pytest.raises(ChfsiError) as ei:
                ctx.apply(X, Z, prec="bf16x3")
            assert ei.value.status == 7
        finally:
            ctx.debug_withhold_arrival(False)
        ctx.apply(X, Z, prec="bf16x3")
        assert torch.equal(Y, Z)
    finally:
        ctx.destroy()
