"""FP32 leaves of an adaptive tree on the GPU whose passes of 32 targets several blocks share (few,
large leaves: launch_rules.h, leaf_a_split) against the same problem as a member of a forest with so
many leaves that one block takes each: the same arithmetic in the same order, bit for bit.  Sizes
leave a partial last pass, fewer and more passes than blocks, an empty problem, and (max_leaf < n) trees
with M2P, L2P and leaves of every size."""
import numpy as np
import pytest
import torch

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def solve(ctx, x, q, offs, s, p, precision):
    n = len(q)
    f = ctx.build_forest(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), np.asarray(offs), max_leaf=s)
    phi = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    E = torch.full((n, 3), np.nan, dtype=torch.float64, device="cuda")
    f.eval(p, phi, E, precision=precision)
    B.dafmm_sync(ctx.h)
    f.free()
    return phi.cpu().numpy(), E.cpu().numpy()


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("n,s,p", [(33, 64, 2), (97, 128, 4), (256, 256, 3), (257, 512, 3), (1000, 1024, 4), (3001, 512, 6),
                                   (2500, 70, 5)])
def test_shared_passes(ctx, n, s, p, precision):
    rng = np.random.default_rng(n)
    x, q = rng.standard_normal((n, 3)), rng.uniform(-1.0, 1.0, n)
    phi, E = solve(ctx, x, q, [0, n], s, p, precision)
    k = 4000  # one-leaf problems around it, the first one empty
    few = rng.standard_normal((2 * k, 3))
    xs, qs = np.concatenate([few[:k], x, few[k:]]), np.concatenate([np.ones(k), q, np.ones(k)])
    offs = np.concatenate([[0], np.arange(0, k + 1, 2), k + n + np.arange(0, k + 1, 2)])
    fphi, fE = solve(ctx, xs, qs, offs, s, p, precision)
    assert np.isfinite(fphi).all() and np.isfinite(fE).all()
    assert np.array_equal(fphi[k:k + n], phi) and np.array_equal(fE[k:k + n], E)
