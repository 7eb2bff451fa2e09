"""Handles may be used from several host threads, and the launchers keep what
they ask the runtime once per device (attributes, occupancy, the driver's
entry point) in function-local statics.  A plain one is a data race whose
outcome no run can be made to show, so the rule is held to the source: such a
static is const (initialised once, by the language's own lock) or atomic.
"""
from __future__ import annotations

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_13359_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_statics_are_const_or_atomic(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    for m in re.finditer(r"^[ \t]+static\s+(?!_assert)([^;={(]*)[;={(]", text, re.M):
        what = m.group(1)
        if m.group(0).endswith("("):  # a member function
            continue
        assert re.match(r"(const|constexpr|std::atomic<)", what.strip()), (os.path.basename(path), what.strip())
