"""Calls that follow one another in a stream without a wait in between.

Every launch may be set up while the one before it still runs, so a chain of
calls that each read what the call before wrote (sample, refine, sample ...,
with torch kernels in between) has to give the bits of the same chain with a
wait after every call; and the same chain captured in a CUDA graph and
replayed gives them too.
"""
import numpy as np
import pytest
import torch

import paper_1408_6373_gb300 as cg

pytestmark = pytest.mark.gpu


def _chain(ctx, g, N, n, steps, wait, state):
    edges, S1, S2, H = state
    for j in range(steps):
        S1.zero_()
        S2.zero_()
        H.zero_()
        wait()
        ctx.sample(g, N, edges, 1 + j * n, n, 0, S1, S2, H)
        wait()
        ctx.refine(g.ndim, N, H, edges)
        wait()


def _state(ndim, N, nc):
    e = torch.tensor(np.tile(np.arange(N + 1) / N, (ndim, 1)), device="cuda")
    S1 = torch.zeros(nc, dtype=torch.float64, device="cuda")
    return e, S1, torch.zeros_like(S1), torch.zeros((ndim, N), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [500, 40000, 700000])
def test_unsynchronised_chain_and_graph_give_the_same_bits(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cg.build_library()
    ndim, N, steps = 4, 64, 6
    rng = np.random.default_rng(n)
    g = cg.genz(ndim, [3, 1], 1.0 + 3.0 * rng.random((2, ndim)), rng.random((2, ndim)))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), cg.Context(0, stream=s.cuda_stream) as ctx:
        ref = _state(ndim, N, 2)
        _chain(ctx, g, N, n, steps, s.synchronize, ref)
        got = _state(ndim, N, 2)
        _chain(ctx, g, N, n, steps, lambda: None, got)
        s.synchronize()
        for a, b in zip(ref, got):
            assert torch.equal(a, b)
        rep = _state(ndim, N, 2)
        uniform = rep[0].clone()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            _chain(ctx, g, N, n, steps, lambda: None, rep)
        for _ in range(2):
            rep[0].copy_(uniform)
            graph.replay()
        s.synchronize()
        for a, b in zip(ref, rep):
            assert torch.equal(a, b)
