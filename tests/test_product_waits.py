"""The waits of the merges on the tensor core (blocks and 1x1 pairs), in every order of events (no GPU).

Two teams of warps cut the steps of a reduction into terms in turn, into slots that are used twice at most; two warps multiply them:
each every second step (two sums of the products of high terms), or both every step (as many sums as there is room for).  A wait on
a barrier only tells the phase with one parity from the phase with the other, so it means what it should only where the earlier
phases are known to be over.  The walk below takes the waits from the library, in the order in which the kernel makes them, lets
every warp move whenever its waits allow, lets products end when they like, and looks at what each step finds."""
import pytest

from paper_2301_12187_b200 import dc

MULTIPLIED = 1


def walk(steps, slots, both, warps=1, waits=dc.selftest_product_waits):
    """Visits every reachable state; returns the faults found, ("terms" | "slot" | "stuck", step)."""
    sites = [waits(s, slots) for s in range(steps)]
    passes = lambda phases_over, parity: (phases_over & 1) != parity
    # the steps of an issuing warp, those that it waits for side by side together
    if both:
        turns = [[list(range(s, min(s + 4, steps))) for s in range(0, steps, 4)]] * 2
    else:
        turns = [[[t for t in (s, s + 2) if t < steps] for s in range(odd, steps, 4)] for odd in (0, 1)]
    mine = [[s for turn in warp for s in turn] for warp in turns]
    faults = set()
    # per team the steps that its warps have cut (sorted: which warp is which does not matter); per issuing warp its turn, how many waits of
    # each of the turn's steps it has behind it, and how many of its steps are multiplied
    start = (((0,) * warps,) * 2, tuple((0, (0,) * len(t[0]) if t else ()) for t in turns), (0, 0))
    seen, todo = {start}, [start]
    while todo:
        cut, issue, over = todo.pop()
        has_cut = lambda s: sum(s // 2 < k for k in cut[s & 1])
        multiplied = lambda s: sum(s in mine[w][:over[w]] for w in range(2))
        def phases(what, slot):
            uses = [s for s in (slot, slot + slots) if s < steps]
            return sum(multiplied(s) for s in uses) // (2 if both else 1) if what == MULTIPLIED else sum(has_cut(s) for s in uses) // warps
        moves = []
        for team in range(2):
            for i, k in enumerate(cut[team]):
                s = 2 * k + team
                if s >= steps or not all(passes(phases(what, slot), parity) for what, slot, parity in sites[s][0]):
                    continue
                if s >= slots and multiplied(s - slots) < (2 if both else 1):
                    faults.add(("slot", s))
                team_cut = tuple(sorted(cut[team][:i] + (k + 1,) + cut[team][i + 1:]))
                moves.append(((team_cut, cut[1]) if team == 0 else (cut[0], team_cut), issue, over))
        for w in range(2):
            turn, behind = issue[w]
            issued = sum(len(t) for t in turns[w][:turn])
            if over[w] < issued:
                moves.append((cut, issue, tuple(n + (v == w) for v, n in enumerate(over))))
            if turn >= len(turns[w]):
                continue
            for i, s in enumerate(turns[w][turn]):
                todo_waits = sites[s][1][behind[i]:]
                if not todo_waits or not passes(phases(*todo_waits[0][:2]), todo_waits[0][2]):
                    continue
                here = (turn, behind[:i] + (behind[i] + 1,) + behind[i + 1:])
                if all(n == len(sites[t][1]) for n, t in zip(here[1], turns[w][turn])):
                    faults.update(("terms", t) for t in turns[w][turn] if has_cut(t) < warps)
                    here = (turn + 1, (0,) * len(turns[w][turn + 1]) if turn + 1 < len(turns[w]) else ())
                moves.append((cut, tuple(here if v == w else issue[v] for v in range(2)), over))
        if not moves and any(over[w] < len(mine[w]) for w in range(2)):
            faults.add(("stuck", min(mine[w][over[w]] for w in range(2) if over[w] < len(mine[w]))))
        for m in moves:
            if m not in seen:
                seen.add(m)
                todo.append(m)
    return faults


# every number of slots that 225 KB hold (ten at 80 columns with long reductions, 13 at 48), odd and even, and small ones with every reuse
@pytest.mark.parametrize("steps,slots,both,warps", [
    (12, 11, False, 1), (13, 11, False, 1), (16, 11, False, 1), (12, 10, False, 1), (14, 13, False, 1), (16, 12, False, 1),
    (10, 5, False, 1), (14, 7, False, 1), (12, 6, False, 1), (7, 5, False, 2), (8, 5, False, 2), (7, 4, False, 2),
    (10, 5, True, 1), (8, 4, True, 1), (7, 5, True, 2), (11, 7, True, 1),
])
def test_no_step_is_multiplied_before_its_terms_are_there(steps, slots, both, warps):
    """Nor does one write a slot that is still read; and no warp waits for good."""
    assert not walk(steps, slots, both, warps)


def test_the_walk_finds_a_wait_for_a_second_phase_alone():
    """The walk tells: without the wait for the first use an odd number of slots goes wrong with two sums, an even one does not."""
    def bare(step, slots):
        cut, multiply = dc.selftest_product_waits(step, slots)
        return cut, multiply[-1:]
    assert ("terms", 11) in walk(12, 11, False, waits=bare)
    assert not walk(12, 10, False, waits=bare)
    assert not walk(10, 5, True, waits=bare)
