"""Mixed-precision filters of ragged blocks (widths and leading dimensions that
are not multiples of four, unaligned columns): the steps run on padded copies,
and every column gets the arithmetic it gets in an aligned block, so the results
are the same bits; nothing outside the block is written."""
import pytest
import torch

from paper_1903_10959_gb300 import workloads as W

from gpu_util import gpu_context

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("prec", ["bf16x3", "mixed", "f16x2"])
@pytest.mark.parametrize("n,ld,off", [(1, 1, 0), (3, 5, 1), (77, 77, 0), (130, 132, 2), (131, 140, 4)])
@pytest.mark.parametrize("sites", [0, 3])
def test_ragged_filter(prec, n, ld, off, sites):
    s = W.small_periodic(seed=400 + n, ncell=4, p=4, L=8.0, n_wells=4, n_want=10)
    if sites:
        s.nl_centres = s.centres[:sites].copy()
        s.nl_h = 0.5 + (torch.arange(4 * sites).reshape(sites, 4) / 8.0).numpy()
    ctx = gpu_context(s, block=256)
    try:
        X0 = torch.tensor(W.start_block(9, ctx.ndofs, n), dtype=torch.float32, device=DEV)
        wide = (n + 3) // 4 * 4
        for degree in (5, 8, 9):                      # in place, and on padded copies
            ref = torch.zeros((ctx.ndofs, wide), dtype=torch.float32, device=DEV)
            ref[:, :n] = X0
            ctx.filter(ref, degree, 3.0, 120.0, -2.0, prec=prec)
            buf = torch.full((ctx.ndofs, ld + off + 3), 7.0, dtype=torch.float32, device=DEV)
            X = buf[:, off:off + n]
            X.copy_(X0)
            ctx.filter(X, degree, 3.0, 120.0, -2.0, prec=prec)
            assert torch.equal(X, ref[:, :n])
            assert bool((buf[:, :off] == 7.0).all()) and bool((buf[:, off + n:] == 7.0).all())
    finally:
        ctx.destroy()
