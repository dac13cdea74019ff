"""Dynamic shared memory is declared with the alignment it is accessed with.

A kernel that reads or writes a dynamic shared array 8 or 16 bytes at a time must say
so in the array's declaration: behind static shared data of another size the array is
otherwise only as aligned as its element type.
"""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ELEMENT = {"float": 4, "unsigned": 4, "int": 4, "float2": 8, "double": 8, "float4": 16}
WIDE = {"float2": 8, "int2": 8, "uint2": 8, "double": 8, "float4": 16, "int4": 16, "uint4": 16, "double2": 16}
DECLARED = re.compile(r"extern\s+__shared__\s+(?:__align__\((\d+)\)\s+)?(\w+)\s+(\w+)\[\]")


def too_narrow(text):
    """(array, declared alignment, access width) of each access wider than its array's alignment."""
    out, found = [], list(DECLARED.finditer(text))
    for n, d in enumerate(found):
        align, name = max(int(d[1] or 0), ELEMENT[d[2]]), d[3]
        body = text[d.end():found[n + 1].start() if n + 1 < len(found) else len(text)]
        widths = [WIDE[t] for t in re.findall(r"reinterpret_cast<(?:const )?(\w+)\s*\*>\(" + name + r"\b", body) if t in WIDE]
        widths += [int(w) for w in re.findall(r"__pipeline_memcpy_async\(" + name + r"\b[^;]*,\s*(\d+)\)", body)]
        out += [(name, align, w) for w in widths if w > align]
    return out


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(ROOT, "paper_2110_00328_gb300", "csrc", "*.cu*"))),
                         ids=os.path.basename)
def test_arrays_are_as_aligned_as_their_accesses(path):
    assert too_narrow(open(path).read()) == []


def test_the_rule_sees_a_narrow_array():
    wide = "reinterpret_cast<uint4*>(win);"
    assert too_narrow("extern __shared__ unsigned win[];" + wide) == [("win", 4, 16)]
    assert too_narrow("extern __shared__ __align__(16) unsigned win[];" + wide) == []
