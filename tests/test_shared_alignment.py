"""Shared-memory arrays that a kernel reads or writes 16 bytes at a time have an
alignment of their own, from their type or a declared one, and do not owe it to
the size of what stands before them."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_11246_gb300", "csrc")
SCALAR = r"(?:const\s+)?(?:float|double|u?int(?:8|16|32|64)?_t|int|unsigned(?:\s+long\s+long)?|uint(?:32|64)_t)"
WIDE = r"(?:float4|uint4|int4|double2|ulonglong2)"


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_wide_access_has_declared_alignment(path):
    src = re.sub(r"//[^\n]*", "", open(path).read())
    bad = []
    for names in re.findall(r"__shared__\s+" + SCALAR + r"\s+([^;]+);", src):  # (no __align__ before the type)
        for name in re.findall(r"(\w+)\s*\[", names):
            wide = r"(?:\bld4\(\s*&?|reinterpret_cast<(?:const\s+)?" + WIDE + r"\s*(?:const\s*)?\*>\(\s*&?|cp_async16\(\s*&?)"
            if re.search(wide + name + r"\b", src):
                bad.append(name)
    assert not bad, bad
