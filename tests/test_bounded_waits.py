"""Kernels whose warps wait for one another through mbarriers give every wait a time limit, and every wait's outcome decides
what its warp does next (no GPU needed: this reads the sources)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_19379_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", ["gram_sl.cu", "update_sl.cu", "gram_tc.cu"])
def test_outcomes_are_used(name):
    waits = re.findall(r"[^\n]*\b(?:bar|warp)_wait\([^;{]*[;{]", code(name))
    assert waits
    for w in waits:
        # the drain of copies or MMAs in flight on the way out has nothing left to decide
        assert re.search(r"(!|=|&&|\() *(live = *)?(bar|warp)_wait\(", w) or "abort, false" in w, w


@pytest.mark.parametrize("name", ["gram_sl.cu", "update_sl.cu", "gram_tc.cu", "sliced.cuh", "tc_ptx.cuh"])
def test_no_handover_without_a_limit(name):
    """bar.arrive hands over to a bar.sync that waits without a limit and miscounts a second arrival."""
    assert "bar.arrive" not in code(name) and "named_arrive" not in code(name)
    if name.endswith(".cu"):
        assert "mbarrier" not in code(name).replace("fence.mbarrier_init", "")  # only through tc_ptx.cuh
