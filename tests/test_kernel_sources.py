"""Orderings that the kernels' sources must show: none of these can be made to fail by running them."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_04359_gb300", "csrc")


def body_of(source, start):
    """The text from the first brace after ``start`` to its match."""
    i = source.index("{", start)
    depth = 0
    for j in range(i, len(source)):
        depth += {"{": 1, "}": -1}.get(source[j], 0)
        if depth == 0:
            return source[i:j + 1]
    raise AssertionError("unbalanced braces")


@pytest.mark.parametrize("name", ["gemm_tc.cu", "gemm_decode_tc.cu", "gemm_dp.cu"])
def test_waiting_warps_are_ordered_after_the_poll(name):
    """One lane polls for another CTA's partial sums and a shuffle hands the outcome to the warp, which orders no memory:
    a fence has to follow it before the other lanes read those sums."""
    with open(os.path.join(CSRC, name)) as f:
        source = f.read()
    body = body_of(source, re.search(r"auto wait_parts = \[&\]", source).end())
    assert "ld_acquire" in body
    assert "__threadfence()" in body[body.rindex("__shfl_sync"):]
