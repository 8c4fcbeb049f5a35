"""Steeply graded adaptive trees on the GPU against the oracle FMM, through the C ABI.

Particles crowd towards one point over twelve octaves, so that neighbouring leaves differ by
many levels: the X lists (P2L) hold leaves of every size, full warps and remainders of
particles, and the box offsets span the whole range of level differences.  Bounds as for the
other adaptive trees: rounding in FP64, 64 u / 160 u (u = 2^-24) in the FP32 paths."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-12, 1e-11), "mixed": (3.8e-6, 1e-5), "fp32": (3.8e-6, 1e-5)}


@pytest.fixture(scope="module")
def ctx():
    B.load()
    c = B.Context(0)
    yield c
    c.close()


def rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / max((b ** 2).sum(), 1e-300)))


def graded(n, seed):
    rng = np.random.default_rng(seed)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    x = 0.37 + 0.3 * d * 2.0 ** (-12.0 * rng.random(n))[:, None]
    return x, rng.uniform(-1.0, 1.0, n)


@pytest.mark.parametrize("p,s,n", [(0, 4, 700), (1, 7, 901), (2, 1, 1200), (4, 33, 4001), (7, 16, 2500), (8, 64, 6007),
                                   (10, 31, 3000)])
def test_graded_tree(ctx, p, s, n):
    x, q = graded(n, 50 + p)
    dom = O.oracle.bounding_cube(x)
    ref_phi, ref_E = O.fmm(x, q, dom, p, max_leaf=s, max_depth=20)
    for prec, (tp, te) in TOL.items():
        tree = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), domain=dom, max_leaf=s)
        phi = torch.empty(n, dtype=torch.float64, device="cuda")
        E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
        tree.eval(p, phi, E, precision=prec)
        B.dafmm_sync(ctx.h)
        tree.free()
        assert rel(phi.cpu().numpy(), ref_phi) <= tp, (prec, rel(phi.cpu().numpy(), ref_phi))
        assert rel(E.cpu().numpy(), ref_E) <= te, (prec, rel(E.cpu().numpy(), ref_E))
