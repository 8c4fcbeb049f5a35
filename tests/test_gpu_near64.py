"""The FP64 near field on the GPU at the sizes where its split of lanes and warps changes, against
the direct sum: one leaf of n particles (passes of 32 lanes down to one, sources shared out over
the other lanes and warps), and uniform trees whose number of leaves selects 8, 2 or 1 warps per
leaf.  Coincident particles, and one pair closer than any power-of-two step, are planted.

A term q / r or q d / r^3 carries a few units u = 2^-53 and a running sum of m terms at most m u of
the sum of their magnitudes: the bound is (m + 16) u of that scale for each target (one leaf).
With a far field the FMM's own error enters: order 10 over a well-separated grid is compared with
the oracle FMM at 1e-12 instead."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def points(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.random((n, 3))
    q = rng.uniform(-1.0, 1.0, n)
    if n >= 4:
        x[1] = x[0]  # coincident
        x[3] = x[2] + np.array([3e-13, -1e-13, 2e-13])
    return x, q


def evaluate(ctx, x, q, p, **kw):
    n = len(q)
    tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=[0.0, 0.0, 0.0, 1.0], **kw)
    phi = torch.empty(n, dtype=torch.float64, device="cuda")
    E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    tree.eval(p, phi, E, precision="fp64")
    B.dafmm_sync(ctx.h)
    tree.free()
    return phi.cpu().numpy(), E.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 4, 7, 13, 16, 25, 26, 31, 32, 33, 49, 63, 97, 300])
@pytest.mark.parametrize("adaptive", [False, True])
def test_one_leaf_direct(ctx, n, adaptive):
    x, q = points(n, 7 + n)
    kw = dict(uniform_depth=-1, max_leaf=max(n, 1)) if adaptive else dict(uniform_depth=0, max_leaf=0)
    phi, E = evaluate(ctx, x, q, 2, **kw)
    L = np.longdouble
    d = x.astype(L)[:, None, :] - x.astype(L)[None, :, :]
    r2 = (d * d).sum(-1)
    far = r2 > 0
    ir = np.where(far, 1 / np.sqrt(np.where(far, r2, 1)), 0)
    tp = q[None, :].astype(L) * ir
    te = (tp * ir * ir)[..., None] * d
    bound = (n + 16) * U
    assert np.all(np.abs(phi - tp.sum(1)) <= bound * np.abs(tp).sum(1))
    scale = np.abs(q[None, :] * (ir * ir).astype(float)).sum(1)
    assert np.all(np.abs(E - te.sum(1)) <= bound * scale[:, None])


@pytest.mark.parametrize("depth,n", [(2, 1500), (3, 6007), (4, 30011)])
def test_warps_per_leaf(ctx, depth, n):
    x, q = points(n, depth)
    rp, rE = O.fmm(x, q, [0.0, 0.0, 0.0, 1.0], 4, uniform_depth=depth)
    phi, E = evaluate(ctx, x, q, 4, uniform_depth=depth, max_leaf=0)
    ok = np.arange(n) > 3  # (the planted pair's huge terms would hide the rest)
    for a, r, tol in ((phi, rp, 1e-12), (E, rE, 1e-11)):
        assert np.sqrt(((a - r)[ok] ** 2).sum() / (r[ok] ** 2).sum()) <= tol
