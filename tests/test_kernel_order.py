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
    text = _source("ubep_sync.cu")
    # strips of payload alone, then those with conditions per word; behind either the buffer may be used again
    _in_order(text, "mine[3 * (b * 32 + lane) + 2] = ", "__syncwarp()", "reinterpret_cast<const uint4*>(mine)[", "__syncwarp()",
              "mine[3 * g + 2] = ", "__syncwarp()", "reinterpret_cast<const uint4*>(mine + ", "__syncwarp()")
    assert text.count("reinterpret_cast<const uint4*>(mine") == 2


def test_a_chunks_cursor_is_reset_before_its_destinations_are_released():
    # (the layout group waits for epoch_bar before it releases pos_flag: what the mover warp stored before it arrived there
    # is ordered in front of that release, what it stores later is not)
    mover = _source("ubep_kernels.cu")
    mover = mover[mover.index("void mover_warp("):mover.index("constexpr int kClusterCountWarps")]
    _in_order(mover, "cursor[x.ch] = 0", "mbar_arrive(x.epoch_bar)")
    assert mover.count("cursor[ch] = 0") + mover.count("cursor[x.ch] = 0") == 1


def test_the_combine_reads_what_its_predecessors_write_with_plain_loads():
    # (it is launched ahead of their end; the read-only path asks for memory that nobody writes while the kernel lives, which
    # the compiler may also assume of const pointers declared __restrict__)
    text = _source("ubep_kernels.cu")
    combine = text[text.index("load_row16(const uint4* a)"):text.index("constexpr int kLayoutThreads")]
    assert "__ldg" not in combine and ".nc." not in combine
    head = combine[combine.index("combine_kernel("):]
    head = head[:head.index("{")]
    assert head.count("__restrict__") == 1 and "uint16_t* __restrict__ out" in head
    _in_order(combine, "griddep_wait();", "slot_pos + ", "load_row16<kStream>")


def test_kernels_launched_ahead_read_with_plain_loads():
    # (a caller's kernel that lets its dependents start early may still be writing the routing table or the replica table)
    for name in ("ubep_common.cuh", "ubep_layout.cuh", "ubep_cluster.cuh", "ubep_few.cuh", "ubep_few.cu", "ubep_kernels.cu"):
        text = _source(name)
        assert "__ldg" not in text and ".nc." not in text, name
