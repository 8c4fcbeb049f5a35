"""Uniform trees of so few particles that one warp takes each FP32 leaf (at most 128 in all:
launch_rules.h, leaf_warps) and of a few more, on the GPU against the oracle FMM; bounds as for every
uniform tree (64 u / 160 u, u = 2^-24; FP64 rounding)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-12, 1e-11), "mixed": (3.8e-6, 1e-5), "fp32": (3.8e-6, 1e-5)}
DOM = [0.0, 0.0, 0.0, 1.0]


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / max((b ** 2).sum(), 1e-300)))


@pytest.mark.parametrize("depth", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 2, 31, 127, 128, 129])
def test_few_particles(ctx, n, depth):
    rng = np.random.default_rng(200 * depth + n)
    x, q = rng.random((n, 3)), rng.uniform(0.5, 1.0, n)
    ref_phi, ref_E = O.fmm(x, q, DOM, 5, uniform_depth=depth)
    for prec, (tp, te) in TOL.items():
        tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=DOM, uniform_depth=depth)
        phi = torch.empty(n, dtype=torch.float64, device="cuda")
        E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        tree.eval(5, phi, E, precision=prec)
        B.dafmm_sync(ctx.h)
        tree.free()
        assert rel(phi.cpu().numpy(), ref_phi) <= tp, (prec, rel(phi.cpu().numpy(), ref_phi))
        assert rel(E.cpu().numpy(), ref_E) <= te, (prec, rel(E.cpu().numpy(), ref_E))
