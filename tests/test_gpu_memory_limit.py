"""Calls on a card without room for the scratch of the fast forms (test hook
chfsi_debug_memory_limit): what ran in the memory of the plain forms still runs,
with their results.

Tolerance: 1e-12, as the binary64 tests of overlap and rotation have it.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W

from gpu_util import gpu_context, rel_fro

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_cholgs_without_digit_scratch():
    """Overlap and rotation on the ALUs, and no error text left behind."""
    ctx = Context(4, 8.0, 4)
    try:
        ctx.build()
        n, M = 40, ctx.ndofs
        X0 = W.start_block(3, M, n)
        X = torch.tensor(X0, device=DEV)
        # the overlap, its inverse factor, 64 partial sums and the rotated block
        ctx.debug_memory_limit(ctx.device_bytes() + (2 + 64) * n * n * 8 + M * n * 8 + 256)
        ctx.cholgs(X)
        assert ctx.last_error() == ""
        ref = np.linalg.solve(np.linalg.cholesky(X0.T @ X0), X0.T).T
        assert rel_fro(X.cpu().numpy(), ref) <= 1e-12
    finally:
        ctx.destroy()
