"""Shared arrays that a kernel reads or writes as 16-byte vectors are declared on 16-byte
boundaries: the placement of a plain float array is the compiler's choice, and a vector access
off its boundary is a fault."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_3830_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_shared_arrays_read_as_vectors_are_aligned(path):
    src = open(path).read()
    vector = set(re.findall(r"\*\((?:const )?(?:float4|int4|uint4|double2)\s*\*\)\s*&?\(?\s*(\w+)", src))
    for quals, decl in re.findall(r"^\s*__shared__([^;=]*?)\b(?:float|int|unsigned|uint32_t|double) ([^;]*);", src, re.M):
        names = set(re.findall(r"(\w+)\[", decl)) & vector
        assert not names or "__align__(16)" in quals, (os.path.basename(path), names)
