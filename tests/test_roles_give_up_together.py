"""The bounded waits of the surrogate's warp-specialised kernels end the block.

A wait that runs out must not leave a lane, or a warp, behind at an unbounded
wait: lanes that each decide for themselves can part at the bound, and warps that
have met their condition would stand at a barrier of the group that the others no
longer reach. None of this can be run on a GPU without a copy that never lands, so
the sources are read: single-lane waits only in the copying role (one lane), one
outcome per warp everywhere else, and within the loops over rows only barriers
that every warp of the group reaches whether or not its wait ran out."""
import os
import re

import pytest

from paper_2106_01557_gb300 import build


def _source(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _copying_role(src):
    """The text of warp 0's role, whose work is a single lane's."""
    a = src.index("if (warp == 0) {")
    role = src[a:src.index("} else if (warp == 1)", a)]
    assert "lane == 0" in role[:role.index("for (")]
    return role


@pytest.mark.parametrize("name", ["lbm_conv_tc.cu", "lbm_wgrad64.cu"])
def test_waits_of_whole_warps_have_one_outcome(name):
    src = _source(name)
    assert len(re.findall(r"\brole_wait\(", src)) == len(re.findall(r"\brole_wait\(", _copying_role(src)))
    assert "role_wait_warp(" in src


def test_groups_leave_their_rows_together():
    # the epilogue's rows end at a vote that a warp reaches whether or not its waits
    # ran out: a failed wait leaves the do-block before it, not the loop
    src = _source("lbm_conv_tc.cu")
    assert "group_sync(" not in src
    row = src[src.index("bool failed = true;"):src.index("if (group_any(grp, failed)) break;")]
    block = row[row.index("do {"):row.index("} while (false);")]
    assert len(re.findall(r"if \((?:with_res && )?!role_wait_warp\([^;]*\) break;", block)) == row.count("role_wait") == 2
    # the bias warps' only barrier comes after their rows
    src = _source("lbm_wgrad64.cu")
    assert src.count("group_sync(") == 1 and "group_any(" not in src
    role = src[src.index("} else if (warp >= 8) {"):]
    assert "role_wait" not in role[role.index("group_sync("):role.index("bool ok = true;", role.index("group_sync("))]
