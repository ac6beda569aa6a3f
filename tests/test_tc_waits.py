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


@pytest.mark.parametrize("name", ["laps_logreg_mma.cu", "laps_logreg_x3.cu"])
def test_the_copying_warp_always_waits_for_its_copies(name):
    """Also when it issued every chunk itself and another role gave up: the waits for the last chunks stand in no
    condition (the producer's block has no branch after its loop but the one that records the failure)."""
    with open(os.path.join(CSRC, name)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    role = src[src.index("tma_load_2d(dst"):src.index("} else if (warp <= 2) {")]
    after = role[role.index("issued = c + 1;"):]
    assert after.count("if (") == 1 and "if (!ok) atomicExch(&s_fail, 1);" in after
    assert re.search(r"for \(int c = max\(0, issued - \w+\); c < issued; \+\+c\)\s*mbar_wait\(", after)


def test_the_warp_wide_wait_votes():
    with open(os.path.join(CSRC, "laps_tc.cuh")) as f:
        src = f.read()
    body = src[src.index("bool mbar_wait_warp("):]
    assert "return __all_sync(0xffffffffu, mbar_wait(bar, parity, deadline));" in body[:body.index("}")]
