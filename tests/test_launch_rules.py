"""How launches split their work (launch_rules.h), on the host."""
import ctypes
import os
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    d = tempfile.mkdtemp(prefix="dafmm_rules_")
    so = os.path.join(d, "rules.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared",
                           "-I", os.path.join(ROOT, "paper_2508_02626_gb300", "csrc"),
                           "-o", so, os.path.join(ROOT, "tests", "launch_rules_check.cpp")])
    h = ctypes.CDLL(so)
    h.bbox_blocks.argtypes = [ctypes.c_longlong, ctypes.c_longlong]
    return h


@pytest.mark.parametrize("nroots", [1, 64, 2000, 20_000, 100_000, 1_000_000])
@pytest.mark.parametrize("max_n", [0, 1, 255, 4097, 1_000_000, 2_000_000_000])
def test_bounding_boxes(lib, nroots, max_n):
    """The empty blocks (0.5 ns each) never cost more than one block per problem would take for the
    largest (2.2 ns a particle), and one problem alone gets all the blocks that it fills."""
    b = lib.bbox_blocks(nroots, max_n)
    assert 1 <= b <= 608
    assert b == 1 or 0.5 * nroots * (b - 1) <= 2.2 * max_n
    if nroots == 1 and max_n:
        assert b == min(608, (max_n + 2047) // 2048)
