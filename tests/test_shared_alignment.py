"""Shared arrays that a kernel reads or writes through a wider vector type
declare that type's alignment (a misaligned vector access is a device fault,
and an array's own element type only promises its own)."""
import os
import re

import pytest

import paper_2306_09257_gb300

CSRC = os.path.join(os.path.dirname(paper_2306_09257_gb300.__file__), "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
SIZE = {"float": 4, "int": 4, "float2": 8, "double": 8, "double2": 16, "float4": 16, "uint2": 8, "uint4": 16}
DECLARED = re.compile(r"__shared__\s+(__align__\((\d+)\)\s+)?(\w+)\s+([^;]+);")
CAST = re.compile(r"reinterpret_cast<\s*(?:const\s+)?(\w+)\s*\*>\(\s*&?\s*(\w+)")


def misaligned(text):
    bad = []
    for kernel in re.split(r"(?=__global__)", text):
        cast = {}
        for vector, name in CAST.findall(kernel):
            cast[name] = max(cast.get(name, 1), SIZE.get(vector, 1))
        for _, align, element, names in DECLARED.findall(kernel):
            for name in re.findall(r"(\w+)\s*\[", re.sub(r"\[[^\]]*\]", "[", names)):
                if cast.get(name, 1) > max(int(align or 1), SIZE.get(element, 1)):
                    bad.append(name)
    return bad


def test_finds_a_missing_alignment():
    body = "__global__ void k() {{ __shared__ {}float a[64][8], b[4]; *reinterpret_cast<float4 *>(&a[1][0]); }}"
    assert misaligned(body.format("")) == ["a"]
    assert misaligned(body.format("__align__(16) ")) == []


@pytest.mark.parametrize("name", SOURCES)
def test_declared_alignment(name):
    with open(os.path.join(CSRC, name)) as f:
        assert misaligned(f.read()) == []
