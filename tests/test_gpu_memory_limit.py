"""Calls on a card without room for the scratch of the fast forms (test hook
chfsi_debug_memory_limit): what ran in the memory of the plain forms still runs,
with their results.

Tolerance: 1e-12, as the binary64 tests of overlap and rotation have it.
"""
import numpy as np
import pytest
import torch

from paper_1903_10959_gb300 import Batch, Context, workloads as W

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


def work_through(ctx, X0, prec):
    """The calls of a solve, and what they leave."""
    X = X0.clone()
    out = []
    if prec == "fp64":
        b = ctx.bounds(20)
        ctx.filter(X, 4, 8.0, 1.05 * b, -4.0)
        ctx.cholgs(X)
        d = ctx.rayleigh_ritz(X)
        out.append(torch.tensor(d))
    else:
        d, _ = ctx.solve(X, 2, 6, 1.05 * ctx.bounds(20), prec=prec)
        out.append(torch.tensor(d))
    r, _ = ctx.residuals(X, d, prec=prec)
    out.append(torch.tensor(r))
    X64 = X.double()
    Y = torch.empty_like(X64)
    ctx.apply(X64, Y)
    ctx.last_timings()
    out.append((X64.T @ Y).diagonal().cpu())
    return out


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("sites", [0, 3])
def test_solve_in_the_memory_of_the_plain_forms(prec, sites):
    """At the bytes that the ALU forms need, at twice those, and between: the same
    calls run, with the same values (1e-10 of the largest; 1e-4 for the filter of a
    block in BF16x3, whose subspace differs in rounding)."""
    s = W.small_periodic(seed=360, ncell=5, p=4, L=10.0, n_wells=4, n_want=40)
    if sites:
        s.nl_centres = s.centres[:sites].copy()
        s.nl_h = 0.5 + np.arange(4 * sites).reshape(sites, 4) / 8.0
    dt = torch.float64 if prec == "fp64" else torch.float32

    def context():
        c = gpu_context(s)
        c.set_blocking(44, 1)
        return c, torch.tensor(W.start_block(3, c.ndofs, 44), dtype=dt, device=DEV)

    ctx, X0 = context()
    ctx.set_fp64_products("alu")
    ref = work_through(ctx, X0, prec)
    need = ctx.device_bytes()
    ctx.destroy()
    tol = 1e-10 if prec == "fp64" else 1e-4
    for part in (1.0, 1.02, 1.1, 1.3, 1.6, 2.0, 3.0):
        ctx, X0 = context()
        try:
            ctx.debug_memory_limit(int(part * need) + 256)
            got = work_through(ctx, X0, prec)
            assert ctx.device_bytes() <= int(part * need) + 256
            assert ctx.last_error() == ""
            for a, b in zip(got, ref):
                assert float((a - b).abs().max()) <= tol * max(1.0, float(b.abs().max()))
        finally:
            ctx.destroy()


def test_one_wide_block_does_not_turn_the_digit_products_off():
    """A block too wide for its scratch runs on the ALUs; a narrower one that fits
    takes the digit slices, and so do all widths once there is room."""
    s = W.small_periodic(seed=361, ncell=4, p=4, L=8.0, n_wells=4, n_want=10)
    ctx, free = gpu_context(s), gpu_context(s)
    try:
        X = torch.tensor(W.start_block(3, ctx.ndofs, 160), device=DEV)
        Y, A, D = torch.empty_like(X), torch.empty_like(X), torch.empty_like(X)
        free.apply(X[:, :40], D[:, :40])
        need = free.device_bytes()
        free.apply(X, D)
        free.last_timings()
        limit = (need + free.device_bytes()) // 2
        free.set_fp64_products("alu")
        free.apply(X, A)
        free.last_timings()
        ctx.set_blocking(160, 1)
        ctx.debug_memory_limit(limit)
        ctx.apply(X, Y)
        ctx.last_timings()
        assert torch.equal(Y, A)                       # the ALU form took over
        ctx.apply(X[:, :40], Y[:, :40])
        ctx.last_timings()
        assert torch.equal(Y[:, :40], D[:, :40])       # digit slices, the same bits
        ctx.debug_memory_limit(0)
        ctx.autotune(X, prec="fp64")                                # lets go of the scratch and starts over
        ctx.set_blocking(160, 1)
        ctx.apply(X, Y)
        ctx.last_timings()
        assert torch.equal(Y, D)
    finally:
        ctx.destroy()
        free.destroy()


@pytest.mark.parametrize("prec", ["bf16x3", "mixed", "tf32"])
@pytest.mark.parametrize("lanes,n", [(1, 77), (1, 1), (2, 259)])
def test_ragged_filter_without_its_copies(prec, lanes, n):
    """A ragged block filtered in the memory of the steps on the block itself (a
    scratch block and the dense cell blocks, rows as wide as the block), and with
    room for one of the padded copies but not for all: the same bits."""
    s = W.small_periodic(seed=362, ncell=4, p=4, L=8.0, n_wells=4, n_want=10)
    rows = 64 * 125

    def context():
        c = gpu_context(s, block=300)
        c.set_filter_lanes(lanes)
        x = torch.zeros((c.ndofs, 4), dtype=torch.float32, device=DEV)
        c.apply(x, torch.empty_like(x), prec=prec)                 # packs the cell data
        return c, c.device_bytes() - rows * 4 * 4                  # without its dense cell blocks

    ctx, base = context()
    X0 = torch.tensor(W.start_block(3, ctx.ndofs, n), dtype=torch.float32, device=DEV)
    ref = X0.clone()
    ctx.filter(ref, 9, 3.0, 120.0, -2.0, prec=prec)
    need = base + ctx.ndofs * n * 4 + rows * n * 4 + 4096
    pad = ctx.ndofs * (n + 3) * 4
    ctx.destroy()
    for limit in (need, need + pad // 2, need + pad, need + rows * 3 * 4 + pad):
        ctx, _ = context()
        try:
            X = X0.clone()
            ctx.debug_memory_limit(limit)
            ctx.filter(X, 9, 3.0, 120.0, -2.0, prec=prec)
            assert ctx.device_bytes() <= limit and ctx.last_error() == ""
            assert torch.equal(X, ref)
        finally:
            ctx.destroy()


@pytest.mark.parametrize("prec", ["bf16x3", "mixed"])
@pytest.mark.parametrize("degree", [5, 6])
def test_batch_without_padded_copies(prec, degree):
    """Ragged members of a batch, one of them without room for its padded copy: the
    same bits, nothing written outside the blocks."""
    shapes = [(3, 21), (4, 40), (3, 7)]
    out = []
    for limited in (False, True):
        ctxs, X = [], []
        for k, (cells, n) in enumerate(shapes):
            s = W.small_periodic(seed=370 + k, ncell=cells, p=4, L=2.0 * cells, n_wells=3, n_want=10)
            c = gpu_context(s)
            buf = torch.full((c.ndofs, n + 2), 7.0, dtype=torch.float32, device=DEV)
            buf[:, 1:1 + n] = torch.tensor(W.start_block(k, c.ndofs, n), dtype=torch.float32, device=DEV)
            ctxs.append(c)
            X.append(buf)
        batch = Batch(ctxs)
        views = [x[:, 1:1 + n] for x, (_, n) in zip(X, shapes)]
        for r in range(2):                             # the second call replays the graph
            if limited:
                ctxs[1].debug_memory_limit(ctxs[1].device_bytes())
            batch.filter(views, degree, [3.0] * 3, [150.0] * 3, [-2.0] * 3, prec=prec)
        out.append(X)
        batch.destroy()
        for c in ctxs:
            c.destroy()
    for a, b in zip(*out):
        assert torch.equal(a, b)
        assert bool((b[:, 0] == 7.0).all()) and bool((b[:, -1] == 7.0).all())
