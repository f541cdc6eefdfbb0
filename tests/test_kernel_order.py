"""Orderings inside the kernels that no run can show to be missing (the hardware mostly delivers them anyway), held against
the source text: which store or barrier stands in front of which."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_06202_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _in_order(text, *marks):
    at = 0
    for m in marks:
        found = text.find(m, at)
        assert found >= 0, f"{m!r} does not follow"
        at = found + len(m)


def test_a_token_flag_strip_is_complete_before_other_lanes_read_it():
    # (a warp vote brings lanes together but orders no memory)
    _in_order(_source("ubep_sync.cu"), "mine[3 * g + 2] = ", "__syncwarp()", "reinterpret_cast<const uint4*>(mine")
