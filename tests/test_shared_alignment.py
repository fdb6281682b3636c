"""Shared arrays that a kernel reads or writes by wider words than their elements must ask for that alignment:
where the compiler puts a shared variable is otherwise bound by the element's size alone."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_01665_gb300", "csrc")
WIDE = {"int2": 8, "uint2": 8, "float2": 8, "longlong2": 16, "int4": 16, "uint4": 16, "float4": 16}
DECL = re.compile(r"__shared__\s+(?:__align__\((\d+)\)\s+)?(?:unsigned\s+)?(\w+)\s+([^;]+);")


def misaligned(text):
    """(array, alignment asked for, alignment read by) of the shared arrays that are read too wide."""
    bad = []
    for align, elem, names in DECL.findall(text):
        own = max(int(align or 1), WIDE.get(elem, 1))
        for name in re.findall(r"(\w+)\s*\[", names):
            casts = re.findall(r"reinterpret_cast<\s*(?:const\s+)?(\w+)\s*\*\s*>\(\s*" + name + r"\b", text)
            need = max([WIDE.get(c, 1) for c in casts], default=1)
            if need > own:
                bad.append((name, own, need))
    return bad


def test_the_check_finds_a_planted_one():
    assert misaligned("__shared__ int32_t a[8], b[4];\n x = reinterpret_cast<const int4 *>(b)[0];") == [("b", 1, 16)]
    assert misaligned("__shared__ __align__(16) int32_t b[4];\n x = reinterpret_cast<int4 *>(b)[0];") == []


def test_wide_shared_accesses_are_aligned():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    bad = {os.path.basename(f): b for f in files if (b := misaligned(open(f).read()))}
    assert not bad, bad
