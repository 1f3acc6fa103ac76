"""Batched tiles at the edges of the tile rule and of the grid table's staging.

A tile's CTA copies the grid table the refinement staged: two entries at a
time where the class's stride is even, one at a time where it is odd, and row
by row for an integral with fewer bins than its class.  Iteration sizes sit on
both sides of a tile (64 32-point blocks) and of the largest number of tiles.
Each logged iteration is held to the FP32 tolerances against the oracle on the
same grid (the second iteration's grid is the one the batch refined).
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1408_6373_gb300 as cg
from tests.tolerances import check_fp32_iteration

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cg.build_library()
    c = cg.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("ndim", [1, 3, 9])
@pytest.mark.parametrize("bins", [[33], [7, 33], [6, 50], [32, 64], [64]])
def test_iterations_match_oracle(ctx, ndim, bins):
    rng = np.random.default_rng(ndim * 100 + len(bins) + bins[0])
    items = [(N, n) for N in bins for n in (2, 2047, 2049, 65535, 65600)]
    par = [(0.5 + rng.random((1, ndim)), rng.random((1, ndim))) for _ in items]

    def specs(iters):
        return [cg.spec(cg.genz(ndim, [O.GAUSSIAN], a, u), nbins=N, nstart=n, maxeval=iters * n)
                for (N, n), (a, u) in zip(items, par)]

    B1, B2 = ctx.batch(specs(1)), ctx.batch(specs(2))
    B1.run()
    B2.run()
    for i, ((N, n), (a, u)) in enumerate(zip(items, par)):
        p = O.Problem(ndim, [O.GAUSSIAN], a, u, nbins=N, bits=23)
        I, V = B2.log(i, 2)
        for j, edges in enumerate((O.grid_uniform(ndim, N), B1.grid(i))):
            ob = O.sample_bounds(p, edges, 1 + j * n, n)
            check_fp32_iteration(I[j], V[j], ob, n, what=(ndim, N, n, j))
    B1.close()
    B2.close()


def test_rows_beyond_2_to_32_floats(ctx):
    # 1800 integrals of 489 tiles, rows of 5120 floats: 4.5e9 floats of partial
    # rows, and the last integral's (behind them) the same bits as alone
    ndim, N, n = 32, 160, 16000000
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB")
    g = cg.genz(ndim, [O.C0], 0.1 * np.ones((1, ndim)), 0.5 * np.ones((1, ndim)))
    last = cg.spec(cg.genz(ndim, [O.GAUSSIAN], 0.3 * np.ones((1, ndim)), 0.4 * np.ones((1, ndim))), nbins=N,
                   nstart=n, maxeval=n)
    B = ctx.batch([cg.spec(g, nbins=N, nstart=n, maxeval=n)] * 1799 + [last])
    B.run()
    r, grid = B.results()[-1], B.grid(1799)
    B.close()
    A = ctx.batch([last])
    A.run()
    a = A.results()[0]
    assert r.integral[0] == a.integral[0] and r.error[0] == a.error[0]
    assert np.array_equal(A.grid(0), grid)
    A.close()
