"""Batched BF16x3 filters of few work items per SM (tc_bf16_batch_rings) run the ring
kernel, larger and smaller ones the stream kernel: the same products in the same order,
so a system's filtered block has the same bits in a batch of either size.
"""
import pytest
import torch

from paper_1903_10959_gb300 import Batch, ChfsiError, Context

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _context(cells, p):
    c = Context(cells, 2.0 * cells, p, periodic=False)
    c.set_potential_gaussians([[0.9 * cells] * 3, [1.2 * cells] * 3], [1.0, 2.0], [0.8, 1.1])
    c.build()
    return c


def _blocks(ctxs, widths, pad):
    """Blocks of the given widths in rows of width + pad floats."""
    g = torch.Generator(device=DEV).manual_seed(7)
    return [torch.rand((c.ndofs, w + pad), generator=g, dtype=torch.float32, device=DEV)[:, :w]
            for c, w in zip(ctxs, widths)]


def _filter(ctxs, X, degree):
    B = Batch(ctxs)
    try:
        n = len(ctxs)
        B.filter(X, degree, [30.0] * n, [400.0] * n, [-3.0] * n, prec="bf16x3")
    finally:
        B.destroy()


# (p, cells of each system, widths, floats past a row): with 152 SMs the items of the
# first batch (4^3 p = 4: two tiles, 128; 6^3 216; p = 6: two per cell and tile, 250, 250,
# 182; p = 7: three, 192, 192, 243) but the first's are within the ring kernel's range;
# those of the batch of six times as many are past it.
@pytest.mark.parametrize("p,cells,widths,pad", [
    (4, [4], [129], 0), (4, [6], [96], 0), (5, [6], [33], 1), (5, [4, 4], [128, 131], 0),
    (6, [5], [100], 0), (6, [5], [37], 2), (6, [3, 4], [128, 5], 1),
    (7, [4], [128], 0), (7, [4], [61], 3), (7, [3, 3], [60, 129], 0)])
@pytest.mark.parametrize("degree", [1, 4])
def test_same_bits_in_batches_of_either_size(p, cells, widths, pad, degree):
    ctxs = [_context(n, p) for n in cells]
    more = [_context(n, p) for n in cells * 5]
    try:
        X0 = _blocks(ctxs, widths, pad)
        X = [x.clone(memory_format=torch.preserve_format) for x in X0]
        Z = [x.clone() for x in X0]
        _filter(ctxs, X, degree)
        _filter(ctxs + more, Z + [x.clone() for x in X0 * 5], degree)
        for x, z in zip(X, Z):
            assert torch.isfinite(x).all()
            assert torch.equal(x, z)
    finally:
        for c in ctxs + more:
            c.destroy()


def test_timeout_is_reported_to_the_batch():
    ctx = _context(5, 6)
    B = Batch([ctx])
    try:
        X = _blocks([ctx], [100], 0)
        Z = [x.clone() for x in X]
        args = (1, [30.0], [400.0], [-3.0])
        B.filter(X, *args, prec="bf16x3")
        ctx.debug_withhold_arrival(True)
        try:
            with pytest.raises(ChfsiError):
                B.filter([Z[0].clone()], *args, prec="bf16x3")
        finally:
            ctx.debug_withhold_arrival(False)
        B.filter(Z, *args, prec="bf16x3")
        assert torch.equal(X[0], Z[0])
    finally:
        B.destroy()
        ctx.destroy()
