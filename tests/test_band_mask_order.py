"""Order of the band's accesses to memory that lanes and warps share.  A race
between them seldom shows in results, so the source is checked."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _source():
    src = open(os.path.join(ROOT, "paper_2411_12365_gb300", "csrc", "burr_band.cu")).read()
    return re.sub(r"//[^\n]*", "", src)


def test_one_lane_reads_and_replaces_the_stored_mask():
    """Every access to the stored mask of a bucket stands under `lane == 0`."""
    src = _source()
    decl = re.search(r"uint64_t \*om\s*=\s*a\.omask[^;]*;", src)
    assert decl
    body = src[decl.end():src.index("S.tdone", decl.end())]
    uses = [m.start() for m in re.finditer(r"\*om\b", body)]
    assert len(uses) == 2
    for u in uses:
        statement = body[max(body.rfind(c, 0, u) for c in ";{}") + 1:u]
        assert re.match(r"\s*if \(lane == 0\b", statement), statement
    assert len(re.findall(r"\bomask\b", src)) == 3   # declared, used above, and set by the launch


def test_stores_of_empty_slots_are_followed_by_a_warp_barrier():
    """Lanes read slots that others emptied (the masks of a bucket's first slots)."""
    src = _source()
    store = re.search(r"S\.ring\[\(bB \+ o \+ \(uint32_t\)lane\) & kRingMask\]\.key = 0;", src)
    assert store
    assert "__syncwarp();" in src[store.end():src.index("continue;", store.end())]


def test_final_threshold_is_written_before_the_second_half_only():
    """The staging warp reads it while the sweeping warp is in the second half."""
    src = _source()
    writes = [m.start() for m in re.finditer(r"S\.tdone = ", src)]
    assert len(writes) == 1
    assert re.search(r"if \(half == 0\) \{\s*$", src[:writes[0]])
