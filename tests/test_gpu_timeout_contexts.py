"""Bounded device waits of contexts side by side, in the binary64 digit-slice
kernels and in the mixed precisions: a withheld arrival (test hook
chfsi_debug_withhold_arrival) makes the waits of one launch run out after 2 s; the
kernel drains and frees its tensor memory, and the context it ran for, and no
other, reports CHFSI_ERR_TIMEOUT and stays usable.

Tolerances: 1e-13 for a binary64 application against the oracle, as the other
binary64 tests have it; equal bits for the same launches on the same data.
"""
import threading

import pytest
import torch

from paper_1903_10959_gb300 import ChfsiError, Context, workloads as W

from gpu_util import oracle_problem, rel_fro

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TIMEOUT = 7                                          # CHFSI_ERR_TIMEOUT


@pytest.fixture()
def pair():
    """Two contexts of one system, each on its own stream, and a block for them."""
    s = W.small_periodic(seed=330, ncell=3, p=4, L=7.5, n_wells=3, n_want=24)
    ctx = []
    for _ in range(2):
        c = Context(s.ncell, s.L, s.p, stream=torch.cuda.Stream())
        c.set_potential_gaussians(s.centres, s.depths, s.widths)
        c.build()
        ctx.append(c)
    X0 = W.start_block(s.seed, ctx[0].ndofs, 40)
    X = torch.tensor(X0, device=DEV)
    ref = oracle_problem(s).apply_Htilde(X0)
    torch.cuda.synchronize()
    yield ctx[0], ctx[1], X, ref
    torch.cuda.synchronize()
    for c in ctx:
        c.destroy()


def late(call):
    with pytest.raises(ChfsiError) as e:
        call()
    assert e.value.status == TIMEOUT and "timed out" in str(e.value)


CALLS = {
    "cholgs": lambda c, X: c.cholgs(X.clone()),
    "filter": lambda c, X: c.filter(X.clone(), 3, 3.0, 120.0, -2.0),
    "rayleigh_ritz": lambda c, X: c.rayleigh_ritz(X.clone()),
    "last_timings": lambda c, X: c.last_timings(),
    "build": lambda c, X: c.build(),
}


@pytest.mark.parametrize("after", sorted(CALLS))
def test_asynchronous_application(pair, after):
    """The application itself returns; the next call reports it, once, and nobody else."""
    a, b, X, ref = pair
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    b.debug_withhold_arrival(True)
    b.apply(X, Y)
    b.debug_withhold_arrival(False)
    # a context beside it, in calls that synchronise and check while b's word is set
    torch.cuda.synchronize()
    a.cholgs(X.clone())
    a.apply(X, Z)
    a.last_timings()
    assert rel_fro(Z.cpu().numpy(), ref) <= 1e-13
    late(lambda: CALLS[after](b, X))
    b.apply(X, Y)
    b.last_timings()
    assert torch.equal(Y, Z)


def test_running_beside_another_context(pair):
    """The other context's calls synchronise while the wait is still running out."""
    a, b, X, ref = pair
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    a.apply(X, Z)
    b.apply(X, Y)
    a.last_timings(), b.last_timings()
    b.debug_withhold_arrival(True)
    b.apply(X, Y)
    for _ in range(3):
        a.filter(X.clone(), 3, 3.0, 120.0, -2.0)
    b.debug_withhold_arrival(False)
    late(b.last_timings)
    b.last_timings()


@pytest.mark.parametrize("call", ["cholgs", "filter", "rayleigh_ritz"])
def test_synchronous_calls(pair, call):
    """Overlap, cell products and projection: the call that waited reports it, also
    where what it left is not positive definite."""
    a, b, X, ref = pair
    b.debug_withhold_arrival(True)
    try:
        late(lambda: CALLS[call](b, X))
    finally:
        b.debug_withhold_arrival(False)
    CALLS[call](a, X)
    Y = torch.empty_like(X)
    b.apply(X, Y)
    b.last_timings()
    assert rel_fro(Y.cpu().numpy(), ref) <= 1e-13


def test_mixed_precisions_beside_another_context(pair):
    """A BF16x3 application whose wait runs out in one thread; a context in another
    keeps applying 3xTF32 products, which synchronise and check."""
    a, b, X, ref = pair
    x = X.float()
    y, z = torch.empty_like(x), torch.empty_like(x)
    b.apply(x, y, prec="bf16x3")                     # packs the cell data
    a.apply(x, z, prec="mixed")
    raised = []

    def wait_in_vain():
        try:
            b.apply(x, y, prec="bf16x3")
        except ChfsiError as e:
            raised.append(e.status)

    b.debug_withhold_arrival(True)
    t = threading.Thread(target=wait_in_vain)
    try:
        t.start()
        calls = 0
        while t.is_alive():
            a.apply(x, z, prec="mixed")              # no error of the other context's
            calls += 1
    finally:
        t.join()
        b.debug_withhold_arrival(False)
    a.apply(x, z, prec="mixed")
    assert raised == [TIMEOUT] and calls > 10
    b.apply(x, y, prec="bf16x3")
    assert rel_fro(y.double().cpu().numpy(), ref) < 1e-5
    assert rel_fro(z.double().cpu().numpy(), ref) < 1e-5
