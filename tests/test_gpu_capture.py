"""A binary64 application recorded in a CUDA graph: chfsi_apply is asynchronous
and, once a call of the same width has grown its scratch, capturable.

Recording runs nothing, so a capture right after chfsi_build must neither count
the digit words of the new matrices as made (an application outside the graph
would use those of the potential before) nor leave them out of the graph.

Tolerance: the same launches on the same data, 0.
"""
import pytest
import torch

from paper_1903_10959_gb300 import Context, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def system(stream=None):
    s = W.small_periodic(seed=320, ncell=4, p=4, L=8.0, n_wells=4, n_want=10)
    ctx = Context(s.ncell, s.L, s.p, stream=stream)
    ctx.set_potential_gaussians(s.centres, s.depths, s.widths)
    ctx.build()
    return s, ctx


@pytest.mark.parametrize("replay_first", [False, True])
@pytest.mark.parametrize("block", [64, 40])          # one and two column blocks per call
def test_application_recorded_after_a_rebuild(replay_first, block):
    st = torch.cuda.Stream()
    s, ctx = system(st)
    _, other = system()
    try:
        X = torch.tensor(W.start_block(3, ctx.ndofs, 64), device=DEV)
        Y, G, ref = torch.empty_like(X), torch.empty_like(X), torch.empty_like(X)
        torch.cuda.synchronize()
        ctx.set_blocking(block, 1)
        ctx.apply(X, Y)                              # the scratch and the words of the first potential
        for c in (ctx, other):
            c.set_potential_gaussians(s.centres, 1.5 * s.depths, s.widths)
            c.build()
        other.set_blocking(block, 1)
        other.apply(X, ref)
        graph = torch.cuda.CUDAGraph()
        st.synchronize()
        with torch.cuda.graph(graph, stream=st):
            ctx.apply(X, G)
        G.fill_(0.0)
        torch.cuda.synchronize()
        if replay_first:
            graph.replay()
        torch.cuda.synchronize()
        ctx.apply(X, Y)                              # outside the graph
        torch.cuda.synchronize()
        assert torch.equal(Y, ref)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(G, ref)
    finally:
        torch.cuda.synchronize()
        ctx.destroy()
        other.destroy()


def test_bloch_application_recorded_after_a_new_wavevector():
    """The mixed-precision Bloch blocks are packed on first use after set_kpoint."""
    st = torch.cuda.Stream()
    _, ctx = system(st)
    _, other = system()
    try:
        g = torch.Generator(DEV).manual_seed(5)
        X = torch.view_as_complex(torch.randn((ctx.ndofs, 20, 2), device=DEV, generator=g))
        Y, G, ref = torch.empty_like(X), torch.empty_like(X), torch.empty_like(X)
        torch.cuda.synchronize()
        ctx.set_kpoint([0.3, -0.2, 0.1])
        ctx.apply_kpoint_mixed(X, Y)
        for c in (ctx, other):
            c.set_kpoint([-0.1, 0.25, 0.2])
        other.apply_kpoint_mixed(X, ref)
        graph = torch.cuda.CUDAGraph()
        st.synchronize()
        with torch.cuda.graph(graph, stream=st):
            ctx.apply_kpoint_mixed(X, G)
        torch.cuda.synchronize()
        ctx.apply_kpoint_mixed(X, Y)
        torch.cuda.synchronize()
        assert torch.equal(Y, ref)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(G, ref)
    finally:
        torch.cuda.synchronize()
        ctx.destroy()
        other.destroy()
