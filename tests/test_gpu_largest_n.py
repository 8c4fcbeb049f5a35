"""Particle numbers whose FP32 records would not fit an int index are refused before any array is
read (the arrays here hold three particles)."""
import ctypes

import numpy as np
import pytest

from paper_2508_02626_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,depth", [(2 ** 31 - 2, 0), (2 ** 31 - 8 ** 5, 5), (2 ** 31 - 8 ** 7 - 2, 7)])
def test_refused(n, depth):
    lib = B.load()
    x, q, dom = np.zeros((3, 3)), np.zeros(3), np.array([0.0, 0.0, 0.0, 1.0])
    with B.Context(0) as ctx:
        tree = ctypes.c_void_p()
        rc = lib.dafmm_build_tree(ctx.h, x.ctypes.data, q.ctypes.data, n, dom.ctypes.data, depth, 0, None,
                                  ctypes.byref(tree))
        assert rc == B.DAFMM_ERR_INVALID_ARG and not tree.value
        t = ctx.build_tree(x, q, domain=dom, uniform_depth=2)  # the context stays usable
        t.free()
