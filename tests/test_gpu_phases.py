"""Phase times of an adaptive FP64 evaluation on the GPU: the finest level's M2L by itself, as on uniform
trees, and the same results whether phases are timed or not.  A Gaussian point set, whose finest level
holds a small part of the boxes."""
import numpy as np
import pytest
import torch

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rotation", [0, 1])
def test_finest_level(rotation):
    n = 20_000
    rng = np.random.default_rng(3)
    x, q = rng.standard_normal((n, 3)), rng.uniform(-1.0, 1.0, n)
    B.load()
    with B.Context(0) as ctx:
        B.dafmm_set_option(ctx.h, B.DAFMM_OPT_M2L_ROTATION, rotation)
        t = ctx.build_tree(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(), max_leaf=32)
        assert t.info()["depth"] > 3
        out = []
        for profile in (False, True):
            B.dafmm_set_profiling(ctx.h, profile)
            phi = torch.empty(n, dtype=torch.float64, device="cuda")
            E = torch.empty((n, 3), dtype=torch.float64, device="cuda")
            for _ in range(2):
                t.eval(5, phi, E, precision="fp64")
            B.dafmm_sync(ctx.h)
            out.append((phi.cpu().numpy(), E.cpu().numpy()))
        ph = B.dafmm_last_phase_ms(ctx.h)
        t.free()
    assert 0.0 < ph["m2l_finest"] < 0.8 * ph["m2l"]
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
