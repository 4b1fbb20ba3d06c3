"""Row ends of the allocation-free operator, checked in its source without a GPU: a
row's entries are counted unsigned, so a row whose offsets decrease (an end below
zero would be huge) must be made empty where the offsets are loaded, as a signed
count leaves it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_14568_gb300", "csrc")


def test_decreasing_offsets_are_an_empty_row():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "noalloc.cu")).read())
    assert re.search(r"na_row\(unsigned lo, unsigned hi", src)
    load = src[src.index("bhi = __ldg(rp + i + 1);"):]
    load = load[:load.index("__ballot_sync")]
    assert re.search(r"if \(bhi > blo\)[^;]*;\s*else bhi = blo;", load)


def _row_entries(lo, hi):
    """Entries that na_row's unsigned loop visits (first lane, stride one)."""
    lo, hi = lo & 0xffffffff, hi & 0xffffffff
    return 0 if lo >= hi else hi - lo


def test_why_it_matters():
    assert _row_entries(5, 9) == 4 and _row_entries(6, 4) == 0
    assert _row_entries(8, -1) > 1 << 31                     # unclamped: reads far out of range
    for lo, hi in ((8, -1), (6, 4), (3, 3)):
        assert _row_entries(lo, hi if hi > lo else lo) == 0
