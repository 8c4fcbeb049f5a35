"""Offsets into the per-particle and per-box arrays are formed in 64 bits: an int product of a valid
index and the array's width leaves the 31 bits from 7.2e8 particles (xyz, field), 8e7 boxes (27
colleagues) or 2.7e8 boxes (8 children) on, which the entry points accept and the GPU's memory holds.
Read from the sources: every such subscript's index is cast, or declared as a 64-bit variable."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_02626_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
SUBSCRIPT = re.compile(r"\b(xyz|field|ijk|child|colleague)\[\s*(?:3|8|27)\s*\*\s*(\(size_t\)\s*)?([A-Za-z_]\w*(?:\.\w+|\[\w+\])*)")


def int_subscripts(text):
    """Subscripts whose index is neither cast nor, at its nearest declaration before, 64 bits wide."""
    out = []
    for m in SUBSCRIPT.finditer(text):
        if m.group(2):
            continue
        decl = None
        if re.fullmatch(r"\w+", m.group(3)):
            for decl in re.finditer(r"\b(\w+)\s+(?:\w+\s*=[^;(){}]*,\s*)?%s\b\s*(?:=|\)|,)" % m.group(3), text[:m.start()]):
                pass
        if decl is None or decl.group(1) not in ("int64_t", "size_t"):
            out.append(m.group(0))
    return out


def test_the_check_itself():
    assert int_subscripts("const int i = perm[t]; x = xyz[3 * i + 1];") == ["xyz[3 * i"]
    assert int_subscripts("av.child[8 * list[i] + c]") == ["child[8 * list[i]"]
    assert int_subscripts("int64_t i = 0; x = xyz[3 * i]; y = ijk[3 * (size_t)b];") == []


@pytest.mark.parametrize("name", FILES)
def test_no_int_products(name):
    with open(os.path.join(CSRC, name)) as f:
        assert int_subscripts(f.read()) == []
