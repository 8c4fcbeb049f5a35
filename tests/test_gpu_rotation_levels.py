"""The FP64 M2L by rotation on levels of several waves (32768 boxes and more: one target per warp,
launch_rules.h, rot_targets) on the GPU against the oracle FMM, at FP64 rounding; few particles, so
that most boxes are empty and the far field carries the result."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu
DOM = [0.0, 0.0, 0.0, 1.0]


def rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("p", [4, 7])
def test_depth_five(p):
    n = 3001
    rng = np.random.default_rng(p)
    x, q = rng.random((n, 3)), rng.uniform(-1.0, 1.0, n)
    ref_phi, ref_E = O.fmm(x, q, DOM, p, uniform_depth=5)
    B.load()
    with B.Context(0) as ctx:
        tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=DOM, uniform_depth=5)
        phi = torch.empty(n, dtype=torch.float64, device="cuda")
        E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        tree.eval(p, phi, E, precision="fp64")
        B.dafmm_sync(ctx.h)
        tree.free()
    assert rel(phi.cpu().numpy(), ref_phi) <= 1e-12 and rel(E.cpu().numpy(), ref_E) <= 1e-11
