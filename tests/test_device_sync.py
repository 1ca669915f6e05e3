"""Memory order inside a warp, checked in the sources (a missing barrier shows
on a GPU only by chance): a vote or a broadcast that hands on another lane's
decision orders no memory, so wherever lanes go on to read or overwrite what
that decision is about, __syncwarp() follows it at once."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1102_2143_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*", "", f.read())


def test_votes_and_broadcast_decisions_are_followed_by_a_warp_barrier():
    seen = 0
    for name, text in sources():
        for m in re.finditer(r"\b__(?:all|any|ballot|shfl)_sync\(0xffffffffu, (\w+)", text):
            if m.group(1) == "warp_sum":  # a value, not a decision
                continue
            seen += 1
            end = text.index(";", m.end())
            assert re.match(r"\s*__syncwarp\(\);", text[end + 1:]), (name, text[m.start():end + 1])
    assert seen >= 3
