"""__ldg (ld.global.nc) is only for memory that nothing writes while the kernel runs.

The traversals are persistent kernels that write their own scratch, and a load
through the non-coherent path is not ordered by the grid barriers between its
writes and its reads.  Every __ldg of those kernels therefore has to name one
of the graph's own arrays, which no traversal writes.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_4518_gb300", "csrc")
GRAPH_ARRAYS = r"\bp\.(off|adj|toff|tadj|dead|probe|rank)\b"


def ldg_arguments(text):
    for m in re.finditer(r"\b__ldg\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text.count("\n", 0, m.start()) + 1, text[m.end():i - 1]


@pytest.mark.parametrize("name", ["level_loop.cu", "batch.cu", "claims.cuh"])
def test_readonly_loads_name_the_graphs_arrays(name):
    with open(os.path.join(CSRC, name)) as f:
        found = list(ldg_arguments(f.read()))
    bad = [(line, arg) for line, arg in found if not re.search(GRAPH_ARRAYS, arg)]
    assert not bad, f"{name}: __ldg of memory that the kernel may write: {bad}"
    assert found or name == "claims.cuh"
