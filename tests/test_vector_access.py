"""Shared-memory arrays that the kernels read or write through a vector type (float2, int4, ...) state an alignment that
the vector access needs: declared with __align__ of at least its size, or of a vector type that large. Where an
array without one lands is up to the compiler, and a misaligned vector access ends the context. Source text only."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_20043_gb300", "csrc")
SIZE = {"float2": 8, "int2": 8, "uint2": 8, "float4": 16, "int4": 16, "uint4": 16, "double2": 16}
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def misaligned(text):
    """(array, vector type) of every cast of a __shared__ array whose declaration does not align it."""
    shared = {}
    for m in re.finditer(r"__shared__\s+([^;]*);", text):
        decl = m.group(1)
        stated = max([int(a) for a in re.findall(r"__align__\((\d+)\)", decl)] +
                     [SIZE[t] for t in re.findall(r"\b\w+\b", decl) if t in SIZE] + [0])
        for name in re.findall(r"(\w+)\s*\[", decl):
            shared[name] = stated
    casts = re.findall(r"reinterpret_cast<\s*(?:const\s+|volatile\s+)*(\w+)\s*\*\s*>\(\s*&?\s*(\w+)", text)
    return [(name, vec) for vec, name in casts if vec in SIZE and name in shared and shared[name] < SIZE[vec]]


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_shared_arrays_state_the_alignment_of_their_vector_accesses(path):
    with open(path) as f:
        assert misaligned(f.read()) == []


def test_the_check_sees_an_unaligned_array():
    use = "float2 v = *reinterpret_cast<const float2*>(&s_a[w][t]);"
    assert misaligned("__shared__ float s_a[4][32]; " + use) == [("s_a", "float2")]
    assert misaligned("__shared__ __align__(16) float s_a[4][32]; " + use) == []
    assert misaligned("__shared__ float4 s_a[4][8]; " + use) == []
