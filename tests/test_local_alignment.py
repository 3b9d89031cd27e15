"""A local array that CUDA code reads or writes through a vector type must be declared
with that type's alignment: an array of 4-byte elements is only 4-byte aligned by
itself, and a 16-byte access to one that the compiler keeps in memory may fault."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_06234_gb300", "csrc")
VEC = r"(?:int2|int4|uint2|uint4|float2|float4|double2|ulonglong2|longlong2)"
CAST = re.compile(r"reinterpret_cast<(?:const )?" + VEC + r"\s*\*>\((\w+)\)")
SCALAR = r"(?:u?int(?:8|16|32|64)_t|int|unsigned|float|double|__half|__nv_bfloat16)"


def unaligned(src):
    """(array, line) of every local scalar array cast to a vector pointer but declared without an alignment."""
    bad = []
    for m in CAST.finditer(src):
        name = m.group(1)
        # the nearest declaration before the cast
        decl = None
        for d in re.finditer(r"^.*\b" + SCALAR + r"\s+[^;()]*\b" + name + r"\[\w+\][^;()]*;", src[:m.start()], re.M):
            decl = d
        if decl is not None and "__align__" not in decl.group(0):
            bad.append((name, src.count("\n", 0, m.start()) + 1))
    return bad


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_vector_access_to_local_arrays(path):
    with open(path, encoding="utf-8") as fh:
        assert unaligned(fh.read()) == []


def test_the_rule_sees_an_unaligned_array():
    assert unaligned("int32_t a[4], v[4];\n*reinterpret_cast<int4*>(v) = x;\n") == [("v", 2)]
    assert unaligned("__align__(16) int32_t a[4], v[4];\n*reinterpret_cast<int4*>(v) = x;\n") == []
