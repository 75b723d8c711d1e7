"""The .sync.aligned instructions that move data between registers and tensor memory need all 32 lanes of a warp together.
Their callers do some work for some lanes only (cells outside the grid, rows of an accumulator that are not used), so every
helper that holds such an instruction makes the lanes meet before it; a source check, since a warp that is not together there
is undefined and no test may run it."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_01672_gb300", "csrc",
                   "pfnn_umma.cu")


def test_lanes_meet_before_every_tensor_memory_access():
    text = open(SRC).read()
    starts = [m.start() for m in re.finditer(r"^(?:__device__|__global__|template)", text, flags=re.M)]
    at = [m.start() for m in re.finditer(r'"tcgen05\.(?:ld|st)\.sync\.aligned', text)]
    assert len(at) >= 2
    for a in at:
        body = text[max(s for s in starts if s < a):a]
        assert "__syncwarp();" in body, body[:120]


def test_no_lane_leaves_a_loop_between_tensor_memory_accesses():
    text = open(SRC).read()
    loads = [m.end() for m in re.finditer(r"^ +tmem_ld16\(.*$", text, flags=re.M)]
    assert len(loads) >= 4
    for a in loads:
        assert not re.match(r"\s*if \([^)]*\) continue;", text[a:]), text[a - 100:a + 40]
