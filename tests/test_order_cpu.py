"""Statements whose order or operand marks the results rest on and that no run
is sure to show, read from the kernels' source."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2206_05761_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body_of(src, head):
    """The braces' block that follows `head`."""
    i = src.index("{", src.index(head))
    depth = 0
    for k in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[i:k + 1]
    raise AssertionError(head)


def test_the_encode_orders_its_thresholds_before_they_are_read():
    b = body_of(source("kernels.cuh"), "void encode_tile(")
    write = b.index("sthr[w][j][q] = ")
    read = b.index("sthr[w][0]", write)
    between = b[write:read]
    assert "__syncwarp(" in between or "__syncthreads(" in between
