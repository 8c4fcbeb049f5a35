"""1/sqrt of the FP64 near field on the GPU (near64_list in fmm_order.cuh) over the whole range of its
argument: problems of two particles at distance d on the x axis, charge 1, whose potential is
exactly the kernel's 1/sqrt(r^2) of r^2 = fl(d d).  A forest puts thousands of them through one
evaluation, each with its own domain, so that r^2 runs from zero and the denormals to infinity.

Inside the window of the integer test (high words 0x02000000 to 0x7cffffff, 2^-991 <= r^2 < 2^977) the
kernel takes the series rsqrt_series.  Its seed y has 20 explicit significand bits, so that
y y is exact and the residual e = 1 - x y^2 carries one rounding of size 2^-53 |e|; with a seed good to
2^-19, |e| <= 2^-18 and the first term left out is 5/16 e^3 <= 5/16 2^-54.  The result is rounded once
(2^-53): the bound is 2^-53 (1 + 5/32) + 2^-70.  Outside the window CUDA's rsqrt is taken, documented to 1 ulp
(2^-52 at most).  torch.rsqrt, CUDA's as well, is at most the sum of two such errors away.  r^2 = 0 adds
nothing, r^2 = inf adds 1/inf = 0."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu
LO, HI = 2.0 ** -991, 2.0 ** 977


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def inverse_distances(ctx, d):
    """The potential of the first particle of each pair {0, (d, 0, 0)}, as the kernel computes it."""
    m = len(d)
    x = np.zeros((m, 2, 3))
    x[:, 1, 0] = d
    q = np.ones(2 * m)
    f = ctx.build_forest(torch.from_numpy(x.reshape(-1, 3)).cuda(), torch.from_numpy(q).cuda(),
                         np.arange(0, 2 * m + 1, 2), max_leaf=2)
    phi = torch.full((2 * m,), -1.0, dtype=torch.float64, device="cuda")
    f.eval(0, phi, None, precision="fp64")
    B.dafmm_sync(ctx.h)
    f.free()
    p = phi.cpu().numpy().reshape(-1, 2)
    assert np.array_equal(p[:, 0], p[:, 1])
    return p[:, 0]


def rel_error(y, r2):
    """|y sqrt(r2) - 1| to first order, from the exact y^2 r2."""
    return np.array([abs(float(Fraction(a) ** 2 * Fraction(b) - 1)) / 2 for a, b in zip(y.tolist(), r2.tolist())])


def distances():
    rng = np.random.default_rng(5)
    wide = rng.uniform(1.0, 2.0, 4000) * 2.0 ** rng.integers(-495, 488, 4000)
    near_one = np.sqrt(rng.uniform(1.0, 4.0, 2000))  # every significand, both parities of the exponent
    k = np.arange(-200, 201)
    edges = [c * (1.0 + k * 2.0 ** -52) for c in (2.0 ** -495.5, 2.0 ** 488.5)]
    return np.concatenate([wide, near_one] + edges)


def test_series_and_its_window(ctx):
    d = distances()
    r2 = d * d
    inside = (r2 >= LO) & (r2 < HI)
    assert inside.sum() > 6000 and (r2 < LO).any() and (r2 >= HI).any()
    y = inverse_distances(ctx, d)
    err = rel_error(y, r2)
    assert err[inside].max() <= 2.0 ** -53 * (1 + 5 / 32) + 2.0 ** -70
    cuda = torch.rsqrt(torch.from_numpy(r2).cuda()).cpu().numpy()
    assert err[~inside].max() <= 2.0 ** -52 * 1.001
    assert np.all(np.abs(y - cuda) <= 2.0 ** -51 * 1.001 * cuda)


@pytest.mark.parametrize("exponent", [-536, -520, -511, -497, 489, 500, 510])
def test_outside_the_window(ctx, exponent):
    """Denormal r^2 (below 2^-1022) and both far ends: CUDA's rsqrt."""
    d = np.random.default_rng(600 + exponent).uniform(1.0, 2.0, 64) * 2.0 ** exponent
    r2 = d * d
    assert np.all((r2 > 0) & np.isfinite(r2))
    assert rel_error(inverse_distances(ctx, d), r2).max() <= 2.0 ** -52 * 1.001


def test_zero_and_infinite(ctx):
    d = np.array([2.0 ** -540, 0.0, 2.0 ** 512, 2.0 ** 600])  # r^2 = 0, 0, inf, inf
    assert np.array_equal(inverse_distances(ctx, d), np.zeros(4))
