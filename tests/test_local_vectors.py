"""Vector accesses in the kernels go to memory that is aligned for them: an
array that a thread declares without an alignment of its own is only as
aligned as its elements, so no source casts one to a vector pointer."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_15508_gb300", "csrc")
DECL = re.compile(r"\b(?:float|double|int|unsigned)\s+(\w+)\s*\[")
CAST = r"reinterpret_cast<\s*(?:const\s+)?(?:u?int|float|double)[234]\s*\*\s*>\(\s*&?%s\b"


def _scope(text, start):
    """The rest of the block that text[start] stands in."""
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth < 0:
            return text[start:i]
    return text[start:]


def misaligned_casts(text):
    text = re.sub(r"//[^\n]*", "", text)
    found = []
    for decl in DECL.finditer(text):
        statement = re.split(r"[;{}]", text[:decl.start()])[-1]
        if statement.count("(") > statement.count(")"):
            continue  # a parameter
        if "__align__" not in statement and re.search(CAST % decl.group(1), _scope(text, decl.end())):
            found.append(decl.group(1))
    return found


def test_the_check_sees_them():
    bad = "__device__ void f(const float* w) { float a[8]; *reinterpret_cast<float4*>(a + 4) = x; }"
    assert misaligned_casts(bad) == ["a"]
    assert misaligned_casts(bad.replace("float a[8]", "__align__(16) float a[8]")) == []


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_vector_access_to_plain_local_arrays(path):
    with open(path) as f:
        assert misaligned_casts(f.read()) == []
