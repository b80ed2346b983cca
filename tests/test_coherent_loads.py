"""No kernel reads through the read-only path what may be written while it runs.

A programmatic dependent is resident while its predecessor writes its input, and a
persistent kernel reads what it wrote before a grid-wide barrier. The read-only path
(``__ldg``, or ``const __restrict__`` parameters, which the compiler may read so)
promises memory that nobody writes meanwhile. Checked on the sources.
"""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2303_08609_gb300", "csrc")


def sources():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            yield name, re.sub(r"//[^\n]*", "", f.read())


def functions(text):
    """(head, body) of every kernel: from __global__ to the brace that closes it."""
    for m in re.finditer(r"__global__", text):
        start = text.index("{", m.end())
        depth, end = 0, start
        for end in range(start, len(text)):
            depth += (text[end] == "{") - (text[end] == "}")
            if depth == 0:
                break
        yield text[m.start():start], text[start:end]


def test_shared_loaders_and_dependent_kernels():
    # the kernels of noalloc.cu are launched after their predecessor's end and read
    # only their input
    waits = 0
    for name, text in sources():
        if name != "noalloc.cu":
            assert "__ldg" not in text and "ld.global.nc" not in text, name
        for head, body in functions(text):
            if "pdl_wait" in body or "this_grid" in body:
                waits += 1
                assert "__restrict__" not in head and "__ldg" not in body, (name, head)
    assert waits >= 9
