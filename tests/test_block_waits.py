"""The waits of the one-launch block kernel, in every order of events (no GPU).

Two groups of warps take a block's chunks in turn, both write the operand that a third role (the projection) reads, and all
read weights from stages that a fourth refills.  A wait on a barrier only tells the phase with one parity from the phase with the
other, so it means what it should only where the earlier phases are known to be over.  The walk below takes the waits from
the library, in the order in which the kernel makes them, lets every role move whenever its waits allow, lets weights land in any order,
and looks at what each chunk's stencil finds."""
import pytest

from paper_2301_12187_b200 import dc

OPERAND, WEIGHTS = 0, 1
CHUNKS = 12                                      # three rounds of the longest ring


def walk(groups, operands, stages):
    """Visits every reachable state; returns the faults found, ("operand" | "weights" | "stuck", chunk)."""
    sites = [dc.selftest_block_waits(k, operands, stages) for k in range(CHUNKS)]
    passes = lambda phases_over, parity: (phases_over & 1) != parity
    committed = lambda done, barrier: sum(sites[j][0][1] == barrier for j in range(done))
    landed_in = lambda landed, stage: sum(landed >> j & 1 for j in range(stage, CHUNKS, stages))
    faults = set()
    # weights landed (a bit per chunk), chunks projected, per group its chunk and how many of that chunk's waits it has behind it
    start = (0, 0, tuple((g, 0) for g in range(groups)))
    seen, todo = {start}, [start]
    while todo:
        landed, projected, at = todo.pop()
        written = lambda j, at=at: j < at[j % groups][0]         # its stencil is done and has arrived
        moves = []
        # weights: a stage is asked for again when the chunk that used it is projected, in the chunks' order; what is asked for lands in any
        for j in range(min(CHUNKS, projected + stages)):
            if not landed >> j & 1:
                moves.append((landed | 1 << j, projected, at))
        for g, (k, w) in enumerate(at):
            if k >= CHUNKS:
                continue
            what, barrier, parity = sites[k][1][w]
            over = committed(projected, barrier) if what == OPERAND else landed_in(landed, barrier)
            if passes(over, parity):
                here = (k, w + 1)
                if w + 1 == len(sites[k][1]):                    # the stencil begins
                    if projected < k - operands + 1:
                        faults.add(("operand", k))
                    if not landed >> k & 1:
                        faults.add(("weights", k))
                    here = (k + groups, 0)
                moves.append((landed, projected, at[:g] + (here,) + at[g + 1:]))
        if projected < CHUNKS and landed >> projected & 1 and written(projected):
            moves.append((landed, projected + 1, at))
        if not moves and projected < CHUNKS:
            faults.add(("stuck", projected))
        for m in moves:
            if m not in seen:
                seen.add(m)
                todo.append(m)
    return faults


@pytest.mark.parametrize("groups,operands,stages", [(g, o, s) for g in (1, 2) for o in (1, 2) for s in (2, 3, 4)])
def test_no_stencil_runs_ahead_of_what_it_waits_for(groups, operands, stages):
    """Neither writes an operand that is still read nor reads weights that have not landed; and no role waits for good."""
    assert not walk(groups, operands, stages)


def test_projection_and_stencil_name_the_same_phase():
    """Phases of a barrier follow one another: the chunks that use it have alternating parities, beginning with 0."""
    for operands in (1, 2):
        nth = {}
        for k in range(CHUNKS):
            (buffer, barrier, parity), _ = dc.selftest_block_waits(k, operands, 2)
            assert buffer < operands and barrier < 2
            assert parity == nth.get(barrier, 0) & 1
            nth[barrier] = nth.get(barrier, 0) + 1
