"""Pointers into the same array, one of them written through, carry no
__restrict__: the sweeps of the inverse iteration read and write one column."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_07522_gb300", "csrc")


def test_solver_sweeps_do_not_promise_distinct_columns():
    with open(os.path.join(CSRC, "eigen_tridiag.cu")) as f:
        src = f.read()
    body = src[src.index("void tri_forward("):src.index("__global__ void __launch_bounds__(kVecThreads, 1) k_tri_vectors")]
    into_y = re.findall(r"^\s*(.*\*.*)\b\w+ = c\.Y\b", body, re.M)
    assert len(into_y) == 4
    assert not [p for p in into_y if "__restrict__" in p]
