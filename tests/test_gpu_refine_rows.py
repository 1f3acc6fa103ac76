"""The refinement from partial rows, at bin counts with every row split.

An iteration's histogram reaches the refinement as partial rows (one per CTA
of a pass, one per tile of a batch); the bin counts here take vectors of four,
two and one bins, the row groups that fill their buffer furthest (68, 72, 84,
100) and row counts on both sides of 64.

Tolerances.  With e the relative error of a bin's content, an edge moves by at
most 4 e r_mean / r_j (weights r = ((1 - x) / ln(1/x))^1.5, x = h/s, change by
less than 2 e, and so do the prefix sums); the integrand is mild enough for
r_mean <= 2 r_j, so 8 e.  One integral's rows are the same in cv_sample and in
a run, each side adds them to within 2^-22: e = 2^-21 (FP64: 2^-42 on both
sides together, far above 152 additions).  A batch adds the same points in
other groups: at most 16 binary32 additions on the way to a bin on each side
and as much again for the values, e = 2^-18.
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1408_6373_gb300 as cg

pytestmark = pytest.mark.gpu
BINS = [65, 66, 67, 68, 72, 84, 96, 100, 132, 200, 252, 255, 256]
NDIM = 3


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cg.build_library()
    c = cg.Context(0)
    yield c
    c.close()


def _genz(N):
    u = 0.4 + 0.2 * np.random.default_rng(N).random((1, NDIM))
    return cg.genz(NDIM, [O.GAUSSIAN], 1.2 * np.ones((1, NDIM)), u)


def _refined(ctx, g, N, n, flags):
    """cv_refine of the first iteration's histogram, as cv_sample adds it up."""
    e = torch.tensor(O.grid_uniform(NDIM, N), device="cuda")
    S1 = torch.zeros(1, dtype=torch.float64, device="cuda")
    S2, H = torch.zeros_like(S1), torch.zeros((NDIM, N), dtype=torch.float64, device="cuda")
    ctx.sample(g, N, e, 1, n, flags, S1, S2, H)
    ctx.refine(NDIM, N, H, e)
    ctx.synchronize()
    return e.cpu().numpy()


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [3000, 30000, 3000000])
@pytest.mark.parametrize("N", BINS)
def test_one_integral(ctx, N, n, fp64):
    if fp64 and n > 30000:
        n = 300000
    g, flags = _genz(N), cg.FP64 if fp64 else 0
    I = ctx.integral(cg.spec(g, nbins=N, flags=flags, nstart=n, maxeval=n))
    I.reset()
    I.run()
    I.result()
    got = I.grid()
    I.close()
    assert np.max(np.abs(got - _refined(ctx, g, N, n, flags))) <= 8 * 2.0 ** (-42 if fp64 else -21)


def test_batch_and_server(ctx):
    n, iters = 65000, 3
    g = [_genz(N) for N in BINS]

    def specs(j):
        return [cg.spec(gi, nbins=N, nstart=n, maxeval=j * n) for gi, N in zip(g, BINS)]

    B = ctx.batch(specs(1))
    B.run()
    B.results()
    for i, N in enumerate(BINS):
        assert np.max(np.abs(B.grid(i) - _refined(ctx, g[i], N, n, 0))) <= 8 * 2.0 ** -18, N
    B.close()
    # alone and in a mix: the same bits
    B = ctx.batch(specs(iters))
    B.run()
    mix = B.results()
    grids = [B.grid(i) for i in range(len(BINS))]
    B.close()
    srv = ctx.server()
    burst = [srv.wait(i) for i in [srv.submit(sp) for sp in specs(iters)]]
    for i, sp in enumerate(specs(iters)):
        A = ctx.batch([sp])
        A.run()
        r = A.results()[0]
        assert np.array_equal(A.grid(0), grids[i]), BINS[i]
        assert r.integral[0] == mix[i].integral[0] and r.error[0] == mix[i].error[0], BINS[i]
        A.close()
        s = srv.wait(srv.submit(sp))
        assert s.integral[0] == burst[i].integral[0] and s.error[0] == burst[i].error[0], BINS[i]
        v = ctx.vegas(g[i], nbins=BINS[i], nstart=n, nincrease=0, maxeval=iters * n)
        assert abs(v.integral[0] - r.integral[0]) <= 1e-5 * abs(r.integral[0])
    srv.stop()
