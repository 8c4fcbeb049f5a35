"""Uniform trees of few boxes on the GPU against the oracle FMM: the FP32 leaves share a leaf's
source list among 8, 4 or 1 warps, the tensor-core M2L shares a tile's 189 terms out over several
items (depth 2, 3 and 4), the rotation M2L its displacements over several warps.  Sizes leave
empty leaves, single particles and uneven passes; bounds as for every uniform tree (FP64
rounding; 64 u / 160 u, u = 2^-24, in the FP32 paths; float-float as FP64)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-12, 1e-11), "ff": (1e-12, 1e-11), "mixed": (3.8e-6, 1e-5), "fp32": (3.8e-6, 1e-5)}
DOM = [0.0, 0.0, 0.0, 1.0]


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / max((b ** 2).sum(), 1e-300)))


@pytest.mark.parametrize("depth,n,p", [(2, 60, 3), (2, 3001, 4), (2, 5000, 8), (3, 700, 6), (3, 15013, 8), (3, 9001, 10),
                                       (4, 40009, 5), (4, 30011, 9)])
def test_small_uniform_trees(ctx, depth, n, p):
    rng = np.random.default_rng(100 * depth + p)
    x, q = rng.random((n, 3)), rng.uniform(-1.0, 1.0, n)
    ref_phi, ref_E = O.fmm(x, q, DOM, p, uniform_depth=depth)
    for prec, (tp, te) in TOL.items():
        tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=DOM, uniform_depth=depth)
        phi = torch.empty(n, dtype=torch.float64, device="cuda")
        E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        tree.eval(p, phi, E, precision=prec)
        B.dafmm_sync(ctx.h)
        tree.free()
        assert rel(phi.cpu().numpy(), ref_phi) <= tp, (prec, rel(phi.cpu().numpy(), ref_phi))
        assert rel(E.cpu().numpy(), ref_E) <= te, (prec, rel(E.cpu().numpy(), ref_E))
