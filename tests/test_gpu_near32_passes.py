"""FP32 leaves of more than 32 particles on the GPU against the direct sum: such a leaf is worked on
in several passes by one warp, and each pass starts its sums from zero in shared memory after the
warp has read the sums of the pass before.

Single adaptive leaves (no M2P and no far field between two passes), and crowded leaves of a
uniform tree with one warp per leaf (depth 4): all particles in a block of 2 x 2 x 2 adjacent
leaves, so that every pair is a near one.

Bound for each target, u = 2^-24, relative to the sum of the magnitudes of its terms q / r and
q / r^2: offsets in the leaf's frame are rounded at 1.25 u leaf widths per axis, which is up to 22 u of
a distance of 0.1 leaf widths (closer pairs carry the remainders), once in 1 / r and four times in
the field's terms; a partial sum has at most 64 terms; the charge, 1 / r and the products add about
8 u.  22 + 64 + 8 < 96 and 4 * 22 + 64 + 8 < 192."""
import numpy as np
import pytest
import torch

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def check(ctx, x, q, precision, **kw):
    n = len(q)
    tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=[0.0, 0.0, 0.0, 1.0], **kw)
    phi = torch.empty(n, dtype=torch.float64, device="cuda")
    E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    tree.eval(4, phi, E, precision=precision)
    B.dafmm_sync(ctx.h)
    tree.free()
    d = x[:, None, :] - x[None, :, :]
    r2 = (d * d).sum(-1)
    ir = np.where(r2 > 0, 1.0 / np.sqrt(np.where(r2 > 0, r2, 1.0)), 0.0)
    tp = q[None, :] * ir
    te = (tp * ir * ir)[..., None] * d
    assert np.all(np.abs(phi.cpu().numpy() - tp.sum(1)) <= 96 * U * np.abs(tp).sum(1))
    assert np.all(np.abs(E.cpu().numpy() - te.sum(1)) <= 192 * U * (np.abs(tp) * ir).sum(1)[:, None])


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("n", [33, 49, 64, 65, 97, 200])
def test_one_adaptive_leaf(ctx, n, precision):
    rng = np.random.default_rng(n)
    check(ctx, rng.random((n, 3)), rng.uniform(-1.0, 1.0, n), precision, uniform_depth=-1, max_leaf=n)


@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("counts", [(33, 49, 64, 65, 97, 130, 0, 1), (200, 0, 0, 0, 0, 0, 0, 48)])
def test_crowded_uniform_leaves(ctx, counts, precision):
    rng = np.random.default_rng(sum(counts))
    corner = np.array([[i >> 2 & 1, i >> 1 & 1, i & 1] for i in range(8)]) + 6
    x = np.concatenate([(corner[i] + rng.random((c, 3))) / 16 for i, c in enumerate(counts)])
    check(ctx, x, rng.uniform(-1.0, 1.0, len(x)), precision, uniform_depth=4)
