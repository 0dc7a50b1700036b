"""The ring of k_aff_down (csrc/k_lqr.cu): the copying warp's fetches, waits and barriers against the
reads of the warps that hold the rows, step by step.  A copy is complete only once a wait has covered
its group, and between two barriers the two sides run in any order."""
import re
from pathlib import Path

import pytest

SRC = (Path(__file__).parent.parent / "paper_2407_05433_gb300" / "csrc" / "k_lqr.cu").read_text()
RING = int(re.search(r"kAffRing = (\d+);", SRC).group(1))


@pytest.mark.parametrize("steps", [1, 2, 3, RING - 1, RING, RING + 1, 31, 32, 33, 63, 64, 65, 100])
def test_blocks_and_dimensions_are_there_when_they_are_read(steps):
    groups, ring, sdim = [], [None] * RING, [None] * 4
    landed = 0  # copy groups that a wait has covered

    def fetch(slot):
        if len([g for g in groups if g is not None]) < steps:
            stage = len([g for g in groups if g is not None])
            groups.append(stage)
            return slot, stage
        groups.append(None)
        return None

    def wait(in_flight):
        return max(landed, len(groups) - in_flight)

    def done(stage):
        return stage < landed  # group index = stage while stages are left

    for k in range(RING):
        put = fetch(k)
        if put:
            ring[put[0]] = put[1]
    dim = lambda k: k if k < steps else 0  # noqa: E731
    sdim[0], sdim[1] = dim(0), dim(1)
    landed = wait(RING - 2)
    # between barriers 0 and 1 the rows' warps read block 0 as well as block 1
    slot = 0
    dreg = [dim(j) for j in range(32)]
    dnext = [dim(j) for j in range(32, 64)]
    for k in range(steps):
        # what the rows' warps read in this interval, before and after anything the other side does
        reads = ([0] if k == 0 else []) + ([k + 1] if k + 1 < steps else [])
        want = [(s % RING, s) for s in reads]
        assert all(ring[p] == s and done(s) for p, s in want)
        dims = [(0, dim(0))] * (k == 0) + [((k + 1) & 3, dim(k + 1))]
        assert all(sdim[p] == v for p, v in dims)
        if k > 0:
            put = fetch(slot)
            if put:
                ring[put[0]] = put[1]
            slot = (slot + 1) % RING
        if (k + 2) % 32 == 0:
            dreg, dnext = dnext, [dim(k + 34 + j) for j in range(32)]
        sdim[(k + 2) & 3] = dreg[(k + 2) & 31]
        assert all(ring[p] == s for p, s in want) and all(sdim[p] == v for p, v in dims)
        landed = wait(RING - 3)
    assert len([g for g in groups if g is not None]) == steps
