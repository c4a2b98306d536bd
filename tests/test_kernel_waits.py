"""Programmatic dependents reach their wait on every path (read from the kernels' source, no GPU).

A grid's successor is let in when the grid is complete, and its predecessors are only known to be complete
once it has waited for them: a kernel that can leave before cudaGridDependencySynchronize() would let its
successor run beside them.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_11873_gb300", "csrc")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(", text):
            start = text.index("{", text.index(")", m.end()))
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield f"{os.path.basename(path)}:{m.group(1)}", text[start:i]


def test_no_exit_before_the_wait():
    wait = "cudaGridDependencySynchronize()"
    found = {name: body for name, body in kernels() if wait in body}
    assert len(found) > 10 and "gwl_calgrad.cu:k_cal_moments" in found
    early = [name for name, body in found.items() if re.search(r"\breturn\b", body[:body.index(wait)])]
    assert early == []
