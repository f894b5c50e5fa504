"""Bounded waits are left by whole warps: each warp-wide wait decides by a vote, and nothing but the vote's helper
reads the status word (a lane that read it for itself could leave alone and the others' next vote would not end)."""
import os
import re

import pytest

from paper_1002_3028_gb300 import build as B

SOURCES = sorted(f for f in os.listdir(B.CSRC) if f.endswith((".cuh", ".cu")))


def code(name):
    with open(os.path.join(B.CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


@pytest.mark.parametrize("name", SOURCES)
def test_only_the_vote_reads_the_status_word_on_the_device(name):
    reads = re.findall(r"[^\n]*volatile int \*>\([^\n]*", code(name))
    assert all("__any_sync(0xffffffffu" in r for r in reads), reads


def test_every_bounded_wait_uses_the_vote():
    waits = [w for name in SOURCES for w in re.findall(r"it >= spin_limit[^;]*;", code(name))]
    assert len(waits) == 3
    assert all("wait_given_up(p.status)" in w for w in waits), waits
