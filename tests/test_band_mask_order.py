"""The stored mask of a bucket in the segmented band is read and replaced by one
lane.  A race between the lanes of a warp seldom shows in results, so the source
is checked: every access to the mask stands under `lane == 0`."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_one_lane_reads_and_replaces_the_stored_mask():
    src = open(os.path.join(ROOT, "paper_2411_12365_gb300", "csrc", "burr_band.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    decl = re.search(r"uint64_t \*om\s*=\s*a\.omask[^;]*;", src)
    assert decl
    body = src[decl.end():src.index("S.tdone", decl.end())]
    uses = [m.start() for m in re.finditer(r"\*om\b", body)]
    assert len(uses) == 2
    for u in uses:
        statement = body[max(body.rfind(c, 0, u) for c in ";{}") + 1:u]
        assert re.match(r"\s*if \(lane == 0\b", statement), statement
    assert len(re.findall(r"\bomask\b", src)) == 3   # declared, used above, and set by the launch
