"""The cell data formed on the device: the operator of every degree, boundary
condition and quadrature rule against the oracle, and rebuilds on one context.

Tolerance 1e-13 relative for one binary64 application of a random block, as for
the operator itself.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W
from oracle import hamiltonian as oham

from gpu_util import rel_fro

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("p,q,periodic", [(1, 0, True), (1, 16, False), (2, 3, (True, False, True)), (3, 0, False),
                                          (4, 0, True), (5, 5, (False, False, True)), (6, 0, False),
                                          (8, 12, True)])   # the last in two passes over the y pairs
def test_operator_and_rebuild(p, q, periodic):
    n, L = (3 if p < 5 else 2), 5.0
    rng = np.random.default_rng(10 * p + q)
    xyz = L * rng.random((3, 3))
    width = np.array([0.8, 1.0, 2.5])
    ctx = Context(n, L, p, periodic=periodic, quad_points=q)
    try:
        # no wells, then two sets of depths on the same context
        for depth in (np.zeros(0), 1.0 + rng.random(3), np.array([3.0, 0.0, -1.5]))[0 if p < 6 else 1:3 if p < 8 else 2]:
            k = len(depth)
            ctx.set_potential_gaussians(xyz[:k], depth, width[:k])
            ctx.build()
            prob = oham.Problem(n, p, L, periodic,
                                lambda x: oham.gaussian_wells(x, xyz[:k], depth, width[:k], L, periodic), q=q or None)
            X0 = W.start_block(5, prob.ndofs, 5)
            ref = prob.apply_Htilde(X0)
            Y = torch.empty((prob.ndofs, 5), dtype=torch.float64, device=DEV)
            ctx.set_fp64_operator("cells")
            ctx.apply(torch.tensor(X0, device=DEV), Y)
            assert rel_fro(Y.cpu().numpy(), ref) <= 1e-13
            Y32 = torch.empty((prob.ndofs, 5), dtype=torch.float32, device=DEV)
            x32 = X0.astype(np.float32)
            ctx.apply(torch.tensor(x32, device=DEV), Y32, prec="bf16x3")
            assert rel_fro(Y32.cpu().numpy(), prob.apply_Htilde(x32.astype(np.float64))) <= 1e-5
    finally:
        ctx.destroy()
