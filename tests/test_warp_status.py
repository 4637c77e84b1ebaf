"""A bounded wait answers each lane on its own, so a copy that lands while some
lanes of a warp have run out of polls leaves them with different answers.  Where
a kernel branches on the status around full-warp votes, the status has to be
the warp's (mbar_wait_warp), and so has the abort test that ends its loop.
Checked on the sources: making a wait run out for half a warp is nothing to try
on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_13792_gb300", "csrc")


def _function(path, name):
    """The body of the function defined as `name(`, by brace depth."""
    s = open(os.path.join(CSRC, path)).read()
    at = s.index("{", s.index(f"bool {name}("))
    depth = 0
    for k in range(at, len(s)):
        depth += {"{": 1, "}": -1}.get(s[k], 0)
        if depth == 0:
            return s[at:k + 1]
    raise AssertionError(name)


@pytest.mark.parametrize("path,name", [("grav_eval_df.cuh", "df_item"),
                                       ("grav_backward.cu", "bwd_df_item")])
def test_status_that_guards_votes_is_the_warps(path, name):
    body = _function(path, name)
    guarded = re.search(r"if \(warp_live && got\)", body)
    assert guarded, "the loop body no longer branches on the status: adapt this test"
    assert re.search(r"const bool got = mbar_wait_warp\(", body)
    assert "= mbar_wait_bounded(" not in body
    assert re.search(r"if \(__any_sync\(0xffffffffu, \*\(volatile int \*\)&sm\.abort_flag\)\) break;", body)


def test_the_warps_status_is_a_vote():
    s = open(os.path.join(CSRC, "grav_common.cuh")).read()
    assert re.search(r"mbar_wait_warp\([^)]*\)\s*\{\s*return __all_sync\(0xffffffffu, mbar_wait_bounded\(",
                     s)
