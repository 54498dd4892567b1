"""The tensor-core kernels' bounded waits, by reading their source: a wait that a whole warp makes ends
the same in all its lanes.  After a time-out, lanes that went on alone would stay at the warp's next
collective (tcgen05.ld, __syncwarp) while the others wait at the end of the block, which never comes."""
import os
import re

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00733_gb300",
                        "csrc", "net_tc.cu")).read()


def one_lane_blocks(src):
    """Spans of the `if (lane == 0) { .. }` blocks: code of the lane that issues the MMAs."""
    for m in re.finditer(r"if \(lane == 0\) \{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.start(), i


def test_waits_of_a_warp_end_the_same_in_every_lane():
    spans = list(one_lane_blocks(SRC))
    waits = list(re.finditer(r"ok = [^;]*mbar_wait\([^;]*;", SRC))
    alone = [w for w in waits if any(a < w.start() < b for a, b in spans)]
    warps = [w for w in waits if w not in alone]
    assert len(alone) >= 6 and len(warps) >= 12
    assert all("warp_agrees(" in w.group() for w in warps), [w.group() for w in warps if "warp_agrees(" not in w.group()]
    assert not any("warp_agrees(" in w.group() for w in alone)   # a vote that the other lanes do not join
