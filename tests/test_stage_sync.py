"""Ordering of shared memory in the two-node stage kernel, read from its
source: what a race would look like depends on how the warps are scheduled,
so no run can show that it is absent.

The face pass of a tile writes one slot per lane and the update reads the
slots of other lanes.  Between them stands group_and, for groups of one warp
(p <= 4) and of four.  A warp vote converges the lanes and orders no memory;
__syncwarp and barrier.cta do.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_17917_gb300", "csrc")


def source(name):
    """The file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def braced(text, start):
    """The block that opens at the first brace behind `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_both_forms_of_the_group_vote_order_memory():
    text = source("dg_stage_handoff.cuh")
    body = braced(text, text.index("bool group_and("))
    one_warp = braced(body, body.index("if constexpr (GW == 1)"))
    rest = body[body.index(one_warp) + len(one_warp):]
    assert re.search(r"\b__all_sync\b.*\b__syncwarp\(\)\s*;", one_warp, re.S)
    assert "barrier.cta.red.and" in rest


def test_face_pass_and_update_are_separated_by_it():
    text = source("dg_stage_handoff.cuh")
    write, read = text.index("*slot = to_f4(dH)"), text.index("const float4 *fd = sFD + e * NF;")
    assert write < text.index("group_and<GW>(grp, ok)") < read


def test_a_group_that_gave_up_copies_nothing_more():
    """After a copy wait gave up, the group's mbarrier is a phase behind: in
    the later stages of a fused step a wait on it would return at once and the
    block could end with copies still landing in its shared memory.  So the
    group starts no copy and takes no tile any more."""
    text = source("dg_stage_handoff.cuh")
    issue = braced(text, text.index("auto issue = [&](long long tile)"))
    assert re.search(r"if \([^)]*\bfailed\) return;", issue)
    assert "tile < ntiles && !failed; tile += step, parity ^= 1u" in text
    gave_up = braced(text, text.index("if (!group_and<GW>(grp, ok))"))
    assert re.search(r"\bfailed = true;.*kDrainWaits.*break;", gave_up, re.S)


def test_copies_in_flight_are_waited_for_whatever_the_limit():
    """The limit of dg_set_barrier_limit may be 0.  It bounds the waits of a
    run, not those for copies that would land in a block that has ended."""
    text = source("dg_stage_tc_body.inc")
    drains = [braced(text, text.index("if (failed && tid == 0)")),
              braced(text, text.index("auto copy_wait_failed"))]
    for d, n in zip(drains, (1, 2)):
        assert d.count("kDrainWaits") == n and "bar_limit" not in d
