"""Shared arrays that are read or written in wider pieces than their element type say so in their declaration:
what the compiler places in front of them may change with any other variable of the kernel."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")
WIDTH = {"float2": 8, "uint2": 8, "float4": 16, "uint4": 16}


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_wide_accesses_of_shared_arrays_are_aligned_by_declaration(path):
    source = open(path).read()
    for m in re.finditer(r"(?<!extern )__shared__ ((?:__align__\((\d+)\) )?)(?:float|int32_t|uint32_t|int|__nv_bfloat16) (\w+)\[", source):
        declared, name = int(m.group(2) or 4), m.group(3)
        for use in re.finditer(r"reinterpret_cast<(?:const )?(\w+)\*>\(\s*&?" + name + r"\b", source):
            assert WIDTH.get(use.group(1), 4) <= declared, f"{name} is accessed as {use.group(1)}"
