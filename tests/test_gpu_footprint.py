"""dafmm_footprint against the device memory that builds and first evaluations allocate: a context
whose budget is the estimate takes the tree and evaluates it, in every precision, from device and from
host arrays."""
import numpy as np
import pytest
import torch

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32", "ff"])
@pytest.mark.parametrize("depth,n", [(0, 20), (1, 100), (2, 1500), (3, 8000), (4, 30_000), (-1, 300), (-1, 8000)])
@pytest.mark.parametrize("p", [0, 1, 2, 3, 4, 6, 8, 10])
def test_budget_of_the_estimate(p, depth, n, precision):
    B.load()
    rng = np.random.default_rng(n)
    x, q = rng.random((n, 3)), rng.uniform(-1.0, 1.0, n)
    need = B.dafmm_footprint(n, p, depth, 24, B.PRECISIONS[precision])
    on_device = p % 2 == 0
    if on_device:
        x, q = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
        phi, E = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty((n, 3), dtype=torch.float64, device="cuda")
    else:
        phi, E = np.empty(n), np.empty((n, 3))
    with B.Context(0, hbm_budget_bytes=need) as ctx:
        t = ctx.build_tree(x, q, domain=[0.0, 0.0, 0.0, 1.0], uniform_depth=depth, max_leaf=24)
        t.eval(p, phi, E, precision=precision)
        B.dafmm_sync(ctx.h)
        assert B.dafmm_bytes_in_use(ctx.h) <= need
        t.free()
