"""The refinement's integer arithmetic and the histograms of every bin count.

- cv_refine against the same refinement in numpy's extended precision (long
  double), within 1e-14: the weights carry 2^-55 of
  their scale, their sums are exact, and the logarithm and power behind them
  are good to 2^-49, so an edge is off by less than that over the smallest
  share of a bin these histograms give an edge (~0.1).
- One sampling pass with bin counts on both sides of the histogram's rules (one
  step for N = 2^L >= 32, 32/N steps for smaller powers of two, two to sixteen
  for the others) and FP64 integrands whose products and powers are taken in
  groups, against the oracle.
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1408_6373_gb300 as cg
from tests.tolerances import check_fp32_pass

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cg.build_library()
    c = cg.Context(0)
    yield c
    c.close()


def _refine_ld(H, edges):
    out = edges.copy()
    for d in range(H.shape[0]):
        h, e = H[d].astype(LD), edges[d].astype(LD)
        N = len(h)
        if not np.any(H[d]):
            continue
        s = np.empty(N, dtype=LD)
        s[1:-1] = (h[:-2] + h[1:-1] + h[2:]) / LD(3)
        s[0], s[-1] = (h[0] + h[1]) / LD(2), (h[-2] + h[-1]) / LD(2)
        x = s / s.sum()
        r = np.zeros(N, dtype=LD)
        for k in range(N):
            if x[k] >= 1:
                r[k] = LD(1)
            elif x[k] > 0:
                q = (LD(1) - x[k]) / (-np.log(x[k]) if x[k] < 0.9 else -np.log1p(x[k] - LD(1)))
                r[k] = q * np.sqrt(q)
        C = np.concatenate([[LD(0)], np.cumsum(r)])
        for m in range(1, N):
            t = LD(m) * C[-1] / LD(N)
            j = max(0, min(N - 1, int(np.searchsorted(C, t, side="right")) - 1))
            out[d, m] = float(e[j] + (e[j + 1] - e[j]) * (t - C[j]) / r[j])
    return out


@pytest.mark.parametrize("N", [2, 3, 7, 16, 31, 32, 33, 50, 64, 100, 128, 255, 256])
def test_refine_matches_extended_precision(ctx, N):
    rng = np.random.default_rng(N)
    x = (np.arange(N) + 0.5) / N
    H = np.stack([
        np.ones(N),                                         # even: the grid stays
        1.0 + rng.random(N),
        np.exp(-((x - 0.3) / 0.25) ** 2),
        np.where(rng.random(N) < 0.3, 0.0, np.exp(rng.uniform(-20, 20, N))) + 1e-12,
        1e-200 * (0.1 + rng.random(N)),
        np.where(np.arange(N) == N // 2, 1.0, 1e-9),        # one bin holds nearly all
        np.zeros(N),                                        # empty: the grid stays
        1e200 * (0.1 + rng.random(N)),
    ])
    w = rng.uniform(0.05, 1.0, H.shape)
    edges = np.concatenate([np.zeros((len(H), 1)), np.cumsum(w, axis=1)], axis=1)
    edges /= edges[:, -1:]
    e = torch.tensor(edges, dtype=torch.float64, device="cuda")
    ctx.refine(len(H), N, torch.tensor(H, dtype=torch.float64, device="cuda"), e)
    ctx.synchronize()
    got = e.cpu().numpy()
    assert np.array_equal(got[0], edges[0]) and np.array_equal(got[6], edges[6])
    assert np.all(np.diff(got, axis=1) > 0)
    assert np.max(np.abs(got - _refine_ld(H, edges))) <= 1e-14


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("nbins", [2, 3, 5, 8, 9, 15, 16, 17, 31, 32, 33, 63, 100, 255])
def test_histogram_of_every_bin_count(ctx, nbins, fp64):
    ndim, start, n = 3, 77, 20011
    rng = np.random.default_rng(nbins)
    a, u = 0.5 + rng.random((1, ndim)), rng.random((1, ndim))
    edges = np.tile(np.arange(nbins + 1) / nbins, (ndim, 1)) ** 1.5
    _pass_check(ctx, [O.GAUSSIAN], a, u, edges, start, n, fp64)


@pytest.mark.parametrize("ndim", [1, 7, 8, 9, 16, 17, 32])
def test_fp64_products_and_powers(ctx, ndim):
    rng = np.random.default_rng(ndim)
    fams = [O.PRODUCT_PEAK, O.CORNER_PEAK, O.GAUSSIAN, O.OSCILLATORY]
    a, u = 0.2 + rng.random((4, ndim)), rng.random((4, ndim))
    edges = np.tile(np.arange(51) / 50, (ndim, 1)) ** 1.2
    _pass_check(ctx, fams, a, u, edges, 1, 5003, True)


def _pass_check(ctx, fams, a, u, edges, start, n, fp64):
    ndim, nbins = edges.shape[0], edges.shape[1] - 1
    p = O.Problem(ndim, fams, a, u, nbins=nbins, bits=52 if fp64 else 23)
    ob = O.sample_bounds(p, edges, start, n)
    nc = len(fams)
    S1 = torch.zeros(nc, dtype=torch.float64, device="cuda")
    S2, H = torch.zeros_like(S1), torch.zeros((ndim, nbins), dtype=torch.float64, device="cuda")
    ctx.sample(cg.genz(ndim, fams, a, u), nbins, torch.tensor(edges, device="cuda"), start, n,
               cg.FP64 if fp64 else 0, S1, S2, H)
    ctx.synchronize()
    S1, S2, H = S1.cpu().numpy(), S2.cpu().numpy(), H.cpu().numpy()
    if not fp64:
        check_fp32_pass(S1, S2, H, ob, n)
        return
    assert np.all(np.abs(S1 - ob.S1) <= 1e-12 * ob.A1)
    assert np.all(np.abs(S2 - ob.S2) <= 1e-12 * ob.S2)
    assert np.all(np.abs(H - ob.H) <= 1e-12 * ob.H.max(axis=1, keepdims=True))


@pytest.mark.parametrize("ndim,nbins,flags", [(8, 256, 0), (12, 256, 0), (12, 256, cg.JIT), (23, 128, 0),
                                              (23, 128, cg.SCRAMBLE), (32, 256, 0)])
@pytest.mark.parametrize("start,n", [(1, 1), (255, 257), (256, 4096), (1000001, 30011)])
def test_axes_owned_by_warps(ctx, ndim, nbins, flags, start, n):
    # (bins and dimensions whose histogram copies do not fit: groups of 256
    # points, ragged at both ends.  f = 1 on the uniform grid: every value is
    # 1, so the sums and the bins are exact counts)
    seed = 11
    a = np.ones((1, ndim))
    edges = np.tile(np.arange(nbins + 1) / nbins, (ndim, 1))
    y = O.point_coords(O.SCRAMBLED if flags & cg.SCRAMBLE else O.SOBOL, seed, ndim, start, n, 23).astype(np.int64)
    count = np.stack([np.bincount((y[d] * nbins) >> 23, minlength=nbins) for d in range(ndim)])
    S1 = torch.zeros(1, dtype=torch.float64, device="cuda")
    S2, H = torch.zeros_like(S1), torch.zeros((ndim, nbins), dtype=torch.float64, device="cuda")
    ctx.sample(cg.genz(ndim, [cg.CONST], a, 0.5 * a), nbins, torch.tensor(edges, device="cuda"), start, n, flags,
               S1, S2, H, seed=seed)
    ctx.synchronize()
    assert S1.item() == n and S2.item() == n
    assert np.array_equal(H.cpu().numpy(), count)
