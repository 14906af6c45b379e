"""CPU check of the kernels that wait for the kernel before them on the device
(griddepcontrol.wait): such a grid may live while its inputs are still written,
so none of its pointers may be const __restrict__, which allows the compiler
the read-only load path and loads above the wait.  Reads the sources; no GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_00185_gb300", "csrc")


def kernels(text):
    """(parameter list, body) of every __global__ function."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__", text):
        start = text.index("{", m.end())
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        yield text[m.end():start], text[start:end]


@pytest.mark.parametrize("name,least", [("d2q37_kernels.cu", 4), ("d2q37_kernels_fp32.cu", 2)])
def test_waiting_kernels_take_no_read_only_pointers(name, least):
    waiting = [head for head, body in kernels(open(os.path.join(CSRC, name)).read()) if "griddepcontrol.wait" in body]
    assert len(waiting) >= least
    for head in waiting:
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head), head
