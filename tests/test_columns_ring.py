"""The ring of the mixed force kernel's columns with several units side by side, as a model
on the CPU (work_cols in csrc/nb_force.cu): kSlots shared-memory slots, a full and an empty
barrier each, eight warps that read one unit of a round, release all of the round's slots
and refill in turn. A warp's releases of one round come from different lanes, so another
warp may see them in any order; those of its next round follow them. A wait tests one parity
bit, as the hardware does, so it also passes while the phase two before the wanted one is
the last complete one. No refill may overtake a warp that has not released the unit it
replaces. Where every warp has seen all copies of a round before it releases any of its
slots, no schedule breaks this; where a warp waits for its own unit's copy only, many do
(the model sees the fault)."""
import random

import pytest

SLOTS, WARPS = 4, 8


class Barrier:
    def __init__(self, need):
        self.need, self.got, self.phase = need, 0, 0    # phase: the incomplete one

    def arrive(self):
        self.got += 1
        if self.got == self.need:
            self.got, self.phase = 0, self.phase + 1

    def passes(self, parity):
        return (self.phase - 1) & 1 == parity & 1


def _warp(me, units, lgnu, all_copies, full, empty, issue, release):
    """One warp's program; yields a condition to wait for, or None."""
    used, turn = 0, 1 << lgnu
    while used < units:
        cnt = min(turn, units - used)
        mine = me * turn // WARPS
        v = used + (mine if mine < cnt else 0)
        yield lambda: full[v % SLOTS].passes(v // SLOTS)
        for u in range(used, used + cnt) if all_copies else ():
            yield lambda: full[u % SLOTS].passes(u // SLOTS)
        release(me, range(used, used + cnt))
        for q in range(cnt):
            w = used + SLOTS + q
            if w % WARPS != me or w >= units:
                continue
            yield lambda: empty[w % SLOTS].passes(w // SLOTS - 1)
            issue(w)
        used += cnt


def _run(rng, units, lgnu, all_copies):
    """True if no refill overtook a reader. (A schedule that goes wrong may also get stuck.)"""
    full, empty = [Barrier(1) for _ in range(SLOTS)], [Barrier(WARPS) for _ in range(SLOTS)]
    copies, sent = [], [[] for _ in range(WARPS)]       # copies in flight; rounds of releases not yet seen
    released = [0] * units
    sound = True

    def issue(w):
        nonlocal sound
        if w >= SLOTS and released[w - SLOTS] != WARPS:
            sound = False
        copies.append(w)

    def release(me, round_):
        for u in round_:
            released[u] += 1
        sent[me].append(list(round_))

    for w in range(min(SLOTS, units)):
        issue(w)
    warps = [_warp(k, units, lgnu, all_copies, full, empty, issue, release) for k in range(WARPS)]
    waits = [next(g, None) for g in warps]
    hurry = [rng.choice((0.05, 0.3, 1.0)) for _ in range(WARPS)]
    late = [rng.choice((0.02, 0.3, 1.0)) for _ in range(SLOTS)]
    idle = 0
    while sound and any(w is not None for w in waits) and idle < 200000:
        idle += 1
        kind = rng.random()
        if kind < 0.3 and copies:
            full[copies.pop(rng.randrange(len(copies))) % SLOTS].arrive()
            idle = 0
        elif kind < 0.6:
            k = rng.randrange(WARPS)
            if sent[k]:
                u = rng.choice(sent[k][0])
                if rng.random() < late[u % SLOTS]:
                    empty[u % SLOTS].arrive()
                    sent[k][0].remove(u)
                    if not sent[k][0]:
                        sent[k].pop(0)
                    idle = 0
        else:
            k = rng.randrange(WARPS)
            if waits[k] is not None and rng.random() < hurry[k] and waits[k]():
                waits[k] = next(warps[k], None)
                idle = 0
    assert not sound or idle < 200000, "stuck"
    return sound


@pytest.mark.parametrize("lgnu", [1, 2])
def test_refills_wait_for_every_reader(lgnu):
    rng = random.Random(17 + lgnu)
    assert all(_run(rng, units, lgnu, True) for units in (5, 8, 30, 47) for _ in range(30))


def test_the_model_sees_the_missing_wait():
    rng = random.Random(3)
    assert not all(_run(rng, 40, 2, False) for _ in range(100))
