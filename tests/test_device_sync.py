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


def test_vectors_that_other_blocks_write_are_not_read_as_constant():
    """The cooperative iterations (FRESH) gather vectors that other blocks of
    the same kernel wrote: the functions on that path hold them in plain
    pointers, and the read-only path is for links or for FRESH = false."""
    text = dict(sources())["stencil.cuh"]
    for fn in ("dslash_site_fresh", "dslash_site_f64", "site_among_zeros", "dslash_site_fx", "stag_colour_of", "stag_site",
               "stag_site_fx4"):
        at = re.search(r"__device__ \w+ (?:SiteAcc<T, KIND>|SiteVec<NC>|\w+) " + fn + r"\(", text).start()
        end = text.find("\ntemplate", at)
        body = text[at:end if end > 0 else None]
        assert not re.search(r"__restrict__ (?:src|aux|v[fb])\b", body), fn
        for m in re.finditer(r"__ldg\((\w+)", body):
            line = body[body.rfind("\n", 0, m.start()):m.start()]
            assert m.group(1) == "U" or "FRESH ?" in line, (fn, line)
        if fn != "dslash_site_fresh":
            plain = re.search(r"\bdslash_site<", body)
            assert not plain or "if constexpr (FRESH) dslash_site_fresh" in body, fn
