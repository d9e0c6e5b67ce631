"""The epilogue warps of the tensor-core kernels leave their pair loops as whole
warps.  A lane that leaves alone (its own wait timed out, its own view of the
abort flag) would leave the other lanes in a full-mask operation, which no time
limit ends; and a lane that skips the rest of a pass would enter the next
.sync.aligned tensor-memory load apart from the others.  A timeout cannot be
brought about without a fault, so the source itself is checked."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_09113_gb300", "csrc")


def _epilogue(name):
    """The statements of the branch of the epilogue warps, without comments."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    start = src.rindex("else if (warp >= 4) {")
    depth, i = 1, src.index("{", start) + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[start:i]


@pytest.mark.parametrize("name", ["assemble_digits.cu", "assemble_tc.cu"])
def test_epilogue_leaves_as_a_warp(name):
    body = _epilogue(name)
    assert not re.search(r"\bmbar_wait\(", body), "a lane's own wait: use mbar_wait_warp"
    for head in re.findall(r"\bfor \([^)]*\)", body):
        assert "s_abort" not in head, "the abort flag is read per lane"
    assert not re.search(r"if \(!(valid|act)\) (continue|break|return)", body), "lanes without a cell skip ahead"


def test_warp_wait_votes():
    src = open(os.path.join(CSRC, "bulk.cuh")).read()
    body = src[src.index("bool mbar_wait_warp("):]
    assert "__all_sync(0xffffffffu, mbar_wait(" in body[:body.index("}")]
