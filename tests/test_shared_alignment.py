"""Shared arrays that a kernel reads or writes through a wider type are declared with that type's alignment: the
compiler is free to place a float array, aligned to 4 bytes, behind an odd number of 8-byte entries, and a 16-byte
access to it would then be misaligned.  Checked on the sources, on CPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc")
SIZE = {"char": 1, "int": 4, "unsigned": 4, "float": 4, "double": 8, "int2": 8, "float2": 8, "float4": 16, "int4": 16,
        "double2": 16, "ulonglong2": 16}
DECL = re.compile(r"__shared__\s+(?:__align__\((\d+)\)\s+)?(?:unsigned\s+)?(\w+)\s+([^;]+);")
CAST = re.compile(r"reinterpret_cast<\s*(?:const\s+)?(\w+)\s*\*\s*>\(")


def kernels(src):
    """Bodies of the __global__ functions (up to the next one), comments removed."""
    src = re.sub(r"//[^\n]*", "", src)
    return re.split(r"\b__global__\b", src)[1:]


def argument(text, start):
    """The text between the parenthesis that ends before `start` and its partner."""
    depth, i = 1, start
    while depth:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
    return text[start:i - 1]


def misaligned(body):
    """(array, alignment, access size) of the wider accesses to shared arrays of a kernel."""
    align, base = {}, {}
    for al, typ, names in DECL.findall(body):
        for n in re.findall(r"(\w+)\s*\[", re.sub(r"\[[^\]]*\]", "[", names)):
            align[n], base[n] = max(int(al or 0), SIZE.get(typ, 16)), n
    # pointers set from an array or from another such pointer; the expression's first name is what it points into
    for name, first in re.findall(r"\*(?:\s*const)?\s+?(\w+)\s*=\s*(?:reinterpret_cast<[^>]*>\()?&?(\w+)", body):
        if first in base:
            base[name] = base[first]
    out = []
    for c in CAST.finditer(body):
        first = re.match(r"&?\s*(\w+)", argument(body, c.end()))
        if first and first.group(1) in base:
            a = base[first.group(1)]
            if SIZE.get(c.group(1), 16) > align[a]:
                out.append((a, align[a], SIZE.get(c.group(1), 16)))
    return out


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_wider_accesses_are_aligned(path):
    found = [x for body in kernels(open(path).read()) for x in misaligned(body)]
    assert not found, f"(array, its alignment, bytes of the access): {found}"


def test_the_check_sees_a_misaligned_access():
    body = """ void k() { __shared__ float2 t[3]; __shared__ float s[4][8]; extern __shared__ double m[];
      float* p = s[w]; double* q = m + 3; double* r = q + 8;
      float4* d = reinterpret_cast<float4*>(p); double2* e = reinterpret_cast<double2*>(r);
      float2* f = reinterpret_cast<float2*>(t); }"""
    assert misaligned(body) == [("s", 4, 16), ("m", 8, 16)]
