"""Bounded waits are left by whole warps: each warp-wide wait decides by a reading of the status word that its lanes
share, a vote or one lane's reading handed to the others (a lane that read it for itself could leave alone and the
others' next vote would not end)."""
import os
import re

import pytest

from paper_1002_3028_gb300 import build as B

SOURCES = sorted(f for f in os.listdir(B.CSRC) if f.endswith((".cuh", ".cu")))


def code(name):
    with open(os.path.join(B.CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


SHARED = ("__any_sync(0xffffffffu", "__shfl_sync(0xffffffffu")


@pytest.mark.parametrize("name", SOURCES)
def test_no_lane_reads_the_status_word_for_itself(name):
    reads = re.findall(r"[^\n]*volatile int \*>\([^\n]*", code(name))
    assert all(any(s in r for s in SHARED) for r in reads), reads


def test_every_bounded_wait_shares_its_reading():
    waits = [w for name in SOURCES for w in re.findall(r"it >= spin_limit[^;]*;", code(name))]
    assert len(waits) == 3
    assert all("wait_given_up(p.status)" in w or SHARED[0] in w for w in waits), waits
