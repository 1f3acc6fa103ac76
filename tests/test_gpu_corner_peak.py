"""FP64 corner peak (1 + sum a x)^-(ndim+1) where the base is negative or zero
(negative parameters, which the FP64 path takes as they are).

Single points of few bits, so that the base is exact: the value is the
correctly rounded power within 2 ulp on either sign, and a zero base gives the
infinity that pow gives.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle as O
import paper_1408_6373_gb300 as cg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cg.build_library()
    c = cg.Context(0)
    yield c
    c.close()


def _value(ctx, ndim, a, index):
    edges = torch.tensor(O.grid_uniform(ndim, 2), device="cuda")
    S1 = torch.zeros(1, dtype=torch.float64, device="cuda")
    S2, H = torch.zeros_like(S1), torch.zeros((ndim, 2), dtype=torch.float64, device="cuda")
    g = cg.genz(ndim, [cg.CORNER_PEAK], a * np.ones((1, ndim)), np.zeros((1, ndim)))
    ctx.sample(g, 2, edges, index, 1, cg.FP64, S1, S2, H)
    ctx.synchronize()
    return S1.item()


@pytest.mark.parametrize("ndim,a", [(15, -1.0), (15, 1.0), (31, -1.0), (2, -3.0)])
def test_power_of_either_sign(ctx, ndim, a):
    for index in range(1, 64, 5):
        y = O.point_coords(O.SOBOL, 0, ndim, index, 1, 52)[:, 0]
        s = 1 + Fraction(a) * sum(Fraction(int(v), 2 ** 52) for v in y)
        if s == 0:
            continue
        want = float(1 / s ** (ndim + 1))
        assert abs(_value(ctx, ndim, a, index) - want) <= 2 * np.spacing(abs(want))


def test_zero_base(ctx):
    # index 1 is x = 1/2: 1 - 2 x = 0, pow(0, -2) = inf
    assert _value(ctx, 1, -2.0, 1) == np.inf
