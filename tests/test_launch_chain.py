"""Kernels that the library's graphs may launch early (programmatic dependent launch) must wait for
their predecessor before anything else."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_13628_gb300", "csrc")


def kernels(text):
    """(header, first statement) of every __global__ function defined in the text."""
    for m in re.finditer(r"__global__", text):
        depth, k = 0, m.start()
        while not (depth == 0 and text[k] in "{;"):
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        if text[k] == "{":
            yield text[m.start():k].strip(), text[k + 1:].split(";", 1)[0].strip()


@pytest.mark.parametrize("name", ["solve.cu", "lockstep.cu", "krylov.cuh", "sine.cuh", "dst.cuh", "freespace.cu",
                                  "precond.cu", "net.cu", "transport.cu"])
def test_every_kernel_waits_first(name):
    with open(os.path.join(CSRC, name)) as f:
        found = list(kernels(f.read()))
    assert found
    for header, first in found:
        assert first == "pdl_wait()", header
