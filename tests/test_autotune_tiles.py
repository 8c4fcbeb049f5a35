"""Autotuner host logic (no GPU): the near-field tiles it times hold the context's default, FP64 has
none to time, and a cache entry of another build of the library is not taken."""
import os
import re

import pytest

from paper_2508_02626_gb300 import _build
from paper_2508_02626_gb300 import autotune as A
from paper_2508_02626_gb300 import binding as B


def test_default_tile_is_a_candidate():
    with open(os.path.join(_build.CSRC, "api_types.h")) as f:
        default = int(re.search(r"int leaf_warps = (\d+);", f.read()).group(1))
    for precision in ("fp32", "mixed", B.DAFMM_FP32, B.DAFMM_MIXED):
        assert default in A.tile_candidates(precision) and A.tile_candidates(precision) == A.LEAF_WARPS


@pytest.mark.parametrize("precision", ["fp64", "ff", B.DAFMM_FP64])
def test_fp64_has_one_tile(precision):
    assert len(A.tile_candidates(precision)) == 1


def test_key_names_the_library():
    mine = A.make_key("GB300", 6, "fp32", 1000, 2)
    assert mine == A.make_key("GB300", 6, "fp32", 1000, 2, library=A.library_stamp())
    assert mine != A.make_key("GB300", 6, "fp32", 1000, 2, library="another")
    assert mine != "GB300|p6|fp32|%s" % A.size_class(1000, 2)  # the key without it
