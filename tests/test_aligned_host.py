"""Source check (no GPU): the resident engines' warp-collective tensor-memory accesses are
.sync.aligned, so after a branch on a thread's own lines or rows the warp is brought together before
the next one.  Walks the vector roles line by line."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1105_5256_gb300", "csrc")
TM = re.compile(r"\b(tm_ld|tm_st<V>|tm_st<double>|tm_wait|tm_wait_st|x_add|x_get|y_add)\(")
BRANCH = re.compile(r"\bif \((act|i < cnt|row < own|q < ext|lfix|rfix|e < ev)\b")
TOGETHER = re.compile(r"__syncwarp\(\)|__syncthreads\(\)|bar_sync\(|bar_arrive\(|_sync\(0x")


@pytest.mark.parametrize("name,role", [("engine_resident.cuh", "res_vector_role("), ("engine_resident_csr.cuh", "csr_vector_role(")])
def test_the_warp_is_together_before_aligned_accesses(name, role):
    text = open(os.path.join(CSRC, name)).read()
    body = text[text.index("void " + role):]
    body = body[:body.index("\n}\n")]
    apart, seen, bad = None, 0, []
    skip = 0                                         # inside a lambda that only defines a helper
    for n, line in enumerate(body.split("\n")):
        code = line.split("//")[0]
        if skip or re.match(r"\s*auto (x_get|x_put|x_add|y_add|put|send|start) = \[&\]", code):
            skip += code.count("{") - code.count("}")
            continue
        if TOGETHER.search(code):
            apart = None
        if TM.search(code):
            seen += 1
            if apart is not None:
                bad.append((n, line.strip(), "after", apart))
        if BRANCH.search(code):
            apart = line.strip()
    assert seen >= 10 and not bad, bad
