"""Every kernel waits for the grid before it before anything else.

The library launches its kernels with the programmatic-stream-serialization
attribute, so a kernel's blocks may run while the grid before them still
does; only griddepcontrol.wait (dq_pdl_enter) makes that grid's writes
visible.  A kernel that reads first is right only as long as what precedes
it happens to be complete, which nothing here can run to show, so the rule
is held to the source: dq_pdl_enter() is the first statement of every
kernel that is launched this way (all but the failure-detection self-test,
which is launched plainly and reads no other kernel's results).
"""
from __future__ import annotations

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_13359_gb300", "csrc")


def kernels(text):
    """(name, body from the opening brace on) of every __global__ function."""
    for m in re.finditer(r"__global__", text):
        head = text[m.end():text.index("{", m.end())]
        name = re.findall(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", head))[0]
        yield name, text[text.index("{", m.end()) + 1:]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_kernels_wait_first(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    for name, body in kernels(text):
        if "selftest" in name:
            assert re.search(name + r"<<<", text), name  # a plain launch
            continue
        assert body.lstrip().startswith("dq_pdl_enter();"), name
