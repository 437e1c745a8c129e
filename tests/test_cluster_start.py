"""Distributed shared memory is touched only after a cluster barrier: a CTA's shared memory exists for its peers once
it has started, which nothing but a barrier of the whole cluster says.  Read from the kernels' source, since an access
too early is a fault that no run can be asked to show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_06864_gb300", "csrc")


def users():
    """(file, text) of every function (closed by a brace in the first column) that addresses a peer's memory."""
    out = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            out += [(name, f) for f in re.split(r"^\}\s*$", text, flags=re.M) if "map_shared_rank(" in f]
    return out


@pytest.mark.parametrize("name,text", users(), ids=lambda v: v if v.endswith((".cu", ".cuh")) else "")
def test_barrier_before_first_access(name, text):
    assert "cl.sync()" in text[:text.index("map_shared_rank(")], name


def test_found():
    assert len(users()) >= 4
