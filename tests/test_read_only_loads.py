"""The persistent batched kernel runs every phase of an iteration in one launch,
so what one phase writes another reads between grid barriers: only the plane
and the pixels' inputs stay as they are.  No pointer of the phases' code may be
declared __restrict__ (or read by __ldg) but the plane's, since either lets the
compiler take the non-coherent path, whose lines outlive a barrier."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_07149_gb300", "csrc")


def read_only(name):
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    return [line.strip() for line in code.splitlines() if "__restrict__" in line or "__ldg" in line or ".nc" in line]


def test_phases_read_no_iteration_state_as_constant():
    assert read_only("scalp_phases.cuh") == []
    assert read_only("scalp_persistent.cu") == []


def test_tile_reads_only_the_plane_as_constant():
    lines = read_only("scalp_assign_tile.cuh")
    assert lines
    for line in lines:
        assert re.search(r"\b(plane|pbox)\b", line), line
