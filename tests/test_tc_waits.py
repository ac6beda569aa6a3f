"""Waits of the tensor-core kernels' warp-wide roles.  A warp that goes on to .sync.aligned
instructions waits as a whole: a lane that reached the deadline alone would leave the others
to run them without it.  Checked in the source, since a wait that runs out in the middle of
a kernel cannot be timed to split a warp."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2601_16696_gb300", "csrc")


@pytest.mark.parametrize("name", ["laps_logreg_mma.cu", "laps_logreg_x3.cu"])
def test_warp_wide_roles_wait_as_one(name):
    with open(os.path.join(CSRC, name)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    start = src.index("} else if (warp <= 2) {")  # the issuing warps; the epilogue's follow
    roles = src[start:src.index("tcgen05.dealloc", start)]
    assert "warp >= EPI_WARP0" in roles
    single = re.findall(r"\bmbar_wait\(bar\(([^()]*)", roles)
    # one lane's wait for what its warp issued, after the others were told to stop
    assert single and all("DRAIN" in s for s in single), single
    assert len(re.findall(r"\bmbar_wait_warp\(", roles)) == 8


def test_the_warp_wide_wait_votes():
    with open(os.path.join(CSRC, "laps_tc.cuh")) as f:
        src = f.read()
    body = src[src.index("bool mbar_wait_warp("):]
    assert "return __all_sync(0xffffffffu, mbar_wait(bar, parity, deadline));" in body[:body.index("}")]
