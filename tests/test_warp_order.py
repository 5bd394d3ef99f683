"""Shared memory that one lane writes and another reads needs a warp barrier in between:
votes and shuffles order no memory.  A missing one cannot be made to show on a GPU at
will, so this reads the source of the selection's ranking step."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_27952_gb300", "csrc")


def test_ranking_orders_the_winners_entries_before_the_bound():
    """A round's best keys go to top_s from whichever lane holds them; lane 0 then reads the
    last entry to merge the bound into it, and every lane reads all of them."""
    with open(os.path.join(CSRC, "select_gram.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    first = src.index("top_s[e] = k1;")
    merge = src.index("top_s[a.mc] = max(top_s[a.mc], bound);", first)
    read = src.index("kk = top_s[e];", merge)
    assert "__syncwarp();" in src[first:merge]
    assert "__syncwarp();" in src[merge:read]
