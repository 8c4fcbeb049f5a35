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
    h.leaf_warps.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    h.leaf_a_split.argtypes = [ctypes.c_longlong, ctypes.c_int]
    h.rot_targets.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    h.rot_share.argtypes = [ctypes.c_longlong, ctypes.c_int]
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


@pytest.mark.parametrize("nleaves", [1, 15, 200, 456, 457, 3648, 3649, 100_000])
@pytest.mark.parametrize("max_leaf", [0, 1, 32, 33, 200, 1000, 1 << 30])
def test_adaptive_leaves(lib, nleaves, max_leaf):
    """Several blocks per leaf only where every one of them has a pass and a place on the GPU, and
    then for every leaf too large for one: a lone warp on it was up to 1.44 times slower."""
    s = lib.leaf_a_split(nleaves, max_leaf)
    passes = -(-max_leaf // 32)
    assert 1 <= s <= max(1, min(8, passes))
    assert s == 1 or nleaves * s <= 24 * 152
    if max_leaf > 32 and nleaves <= 24 * 152 // 2:
        assert s >= 2
    if nleaves == 1:
        assert s == max(1, min(8, passes))


@pytest.mark.parametrize("f64", [0, 1])
def test_uniform_leaves(lib, f64):
    """The numbers of leaves that a uniform tree can have (8^depth, depth 0 to 7) reach both forms of the
    near-field kernels, and the rule gives no other."""
    assert [lib.leaf_warps(8 ** d, 10_000, f64) for d in range(8)] == [8, 8, 8, 8, 1, 1, 1, 1]
    assert {lib.leaf_warps(k, 10_000, f64) for k in range(1, 5000)} == {8, 1}


@pytest.mark.parametrize("depth", [0, 2, 3])
def test_few_particles(lib, depth):
    """At most one segment of 128 sources in all: nothing to share out in FP32 (FP64 shares single
    sources)."""
    assert [lib.leaf_warps(8 ** depth, n, 0) for n in (0, 1, 2, 128, 129, 1000)] == [1, 1, 1, 1, 8, 8]
    assert [lib.leaf_warps(8 ** depth, n, 1) for n in (0, 2, 128, 129)] == [8, 8, 8, 8]


def test_rotation(lib):
    """Levels 2 to 7: two targets per warp between 512 boxes and one wave in FP64 (at 32768 boxes and more
    they were up to 8 % slower than one), from 512 boxes on in float-float, never in the full basis; the
    displacements shared out until the level has 16 warps per SM, or 8 warps per target."""
    nbox = [8 ** l for l in range(2, 8)]
    assert [lib.rot_targets(b, 1, 1) for b in nbox] == [1, 2, 2, 1, 1, 1]
    assert [lib.rot_targets(b, 1, 0) for b in nbox] == [1, 2, 2, 2, 2, 2]
    assert [lib.rot_targets(b, 0, f) for b in nbox for f in (0, 1)] == [1] * 12
    for b in nbox:
        for t in (1, 2):
            k = lib.rot_share(b, t)
            assert k in (1, 2, 4, 8) and (k == 8 or b // t * k >= 2432) and (k == 1 or b // t * (k // 2) < 2432)
