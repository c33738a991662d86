"""The shared entry tables of the paper's gain are written by all lanes of a team
(atomics on shared memory) and then read slot by slot by other lanes.  A warp
vote brings the lanes together but orders none of their memory accesses, so the
function that fills a table has to end with the team's barrier, for teams of
one warp too.  A missing barrier cannot be shown by running the kernel (the
hardware mostly orders the accesses all the same), so the source is read."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03211_gb300", "csrc",
                   "lf_run.cu")


def test_filling_a_table_ends_with_the_teams_barrier():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    start = text.index("bool lit_fill(")
    body = text[start:text.index("\n}\n", start)]
    after = body[body.index("lit_warp_entries<"):]
    # top-level statements of the function (four spaces) after the inserts: the last two
    last = [line.strip() for line in after.split("\n") if re.match(r"    \S", line)][-2:]
    assert last == ["team_sync<T>(tm);", "return ok;"], last
