"""The trust-region solver's threads read the state of the multiplier search
from shared memory while others run ahead.  No result shows a store that a
slower thread's read is not ordered against (it stores the same value), so
the sources are checked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1803_00113_gb300", "csrc")


def _function(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "trsolve.cuh")).read())
    m = re.search(r"static __device__ \w+ %s\([^)]*\)\s*\{" % name, text) or \
        re.search(r"static __device__ __forceinline__ \w+ %s\([^)]*\)\s*\{" % name, text)
    return text[m.end():text.index("\n}", m.end())]


def test_norm_at_zero_is_stored_once_before_it_is_read():
    body = _function("locate32")
    at = body.index("S.loc[2] =")
    assert body.count("S.loc[2] =") == 1
    # not in anything that later rounds of the search run again ...
    for lam in re.finditer(r"auto \w+ = \[&\]", body):
        end = body.index("\n  };", lam.start()) if "\n" in body[lam.start():body.index(";", lam.start())] \
            else body.index(";", lam.start())
        assert not lam.start() < at < end, "stored by every round"
    # ... and read behind the barrier of the round that stores it
    between = body[at:body.index("= S.loc[2]")]
    assert "narrow(" in between or "first_hit(" in between


def test_search_state_is_written_after_every_lane_has_read_it():
    body = _function("tr_solve")
    write = body.index("S.lo = lo;")
    before = body[body.index("lo = S.lo"):write]
    assert re.search(r"__syncwarp\(\);\s*if \(lane == 0\) \{\s*$", before)
