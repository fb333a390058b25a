"""The ring of stages of the split-operand kernel with two issuing warps, searched state by state: whatever the order in which the producer and the
issuers come to run, no stage is freed and filled again before both issuers have seen it full (a barrier's parity would then tell the late one that it
is empty, and the wait would run out)."""
import os
import re

import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_00094_b200", "csrc", "split_conv.cuh")


def stuck_states(stages, arrivals, period, chunks=14):
    """How many reachable states have chunks left and nobody who can go on.  `period` chunks belong to one issuer, the next ones to the other; the commit
    of a chunk's issuer counts as early as it can come."""
    start = (0, (0,) * stages, (0,) * stages, (0,) * stages, (0, 0))     # chunks loaded; per stage: times full, arrivals, times freed; issuers' chunks
    seen, todo, stuck = {start}, [start], 0
    while todo:
        loaded, full, arrived, freed, at = todo.pop()
        after = []
        s = loaded % stages
        if loaded < chunks and freed[s] % 2 != (loaded // stages + 1) % 2:                # a wait passes when the phase of its parity is over
            after.append((loaded + 1, full[:s] + (full[s] + 1,) + full[s + 1:], arrived, freed, at))
        for me in (0, 1):
            s = at[me] % stages
            if at[me] == chunks or full[s] % 2 == at[me] // stages % 2:
                continue
            a, f = list(arrived), list(freed)
            if at[me] // period % 2 == me or arrivals == 2:
                a[s] += 1
                if a[s] == arrivals:
                    a[s], f[s] = 0, f[s] + 1
            after.append((loaded, full, tuple(a), tuple(f), (at[0] + (me == 0), at[1] + (me == 1))))
        stuck += not after and at != (chunks, chunks)
        for state in after:
            if state not in seen:
                seen.add(state)
                todo.append(state)
    return stuck


@pytest.mark.parametrize("period", [1, 2])
def test_two_issuers_share_a_ring_of_stages(period):
    source = open(HEADER).read()
    stages = int(re.search(r"B_STAGES = BN <= 96 \? (\d) : \d;", source)[1])              # of the tiles of 64 and 80 channels
    found = re.search(r"EMPTY_ARRIVALS = TRIPLE \? (\d) : 1;", source)
    assert stuck_states(stages, int(found[1]) if found else 1, period) == 0
    assert stuck_states(stages, 1, period) > 0                                            # the issuer's commit alone is not enough
