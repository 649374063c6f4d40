"""CPU model of the strip chain (sk_chain.cuh): tickets, their order, and the hand-off buffers.

Every strip of a pair is a ticket.  Tickets are sorted by group, then by bucket
nb - 1 - min((S - s) + cols // 50, nb - 1); within a bucket the order is arbitrary.  Warps take
tickets in order and run them a batch of columns at a time: a strip may take batch b once the strip
before it has handed it on, and may write into its buffer once that buffer is free (a pair's buffers
are used in turn, `ring` of them; a group's memory is that of the group before the last).  The model
runs random interleavings of any number of warps and checks that none is ever stuck, that each batch
is still in the buffer when it is read, and that no buffer is written while a strip still reads it.
"""
import random

import pytest

LAG = 50


def tickets(pairs, groups_of, nb, rng):
    """[(pair, strip)] in ticket order and {(pair, strip): place}."""
    keyed = []
    for p, (S, cols) in enumerate(pairs):
        for s in range(S):
            k = (S - s) + cols // LAG
            keyed.append(((groups_of[p], nb - 1 - min(k, nb - 1)), rng.random(), p, s))
    keyed.sort(key=lambda t: (t[0], t[1]))
    order = [(p, s) for _, _, p, s in keyed]
    return order, {t: i for i, t in enumerate(order)}


@pytest.mark.parametrize("seed", range(6))
def test_a_strip_comes_after_the_one_it_depends_on(seed):
    rng = random.Random(seed)
    pairs = [(rng.randint(1, 40), rng.randint(1, 2000)) for _ in range(60)]
    nb = max(S for S, _ in pairs) + max(c for _, c in pairs) // LAG + 1
    groups_of = [rng.randint(0, 3) for _ in pairs]
    order, place = tickets(pairs, groups_of, nb, rng)
    for p, (S, _) in enumerate(pairs):
        for s in range(1, S):
            assert place[p, s] > place[p, s - 1]
    assert all(groups_of[a[0]] <= groups_of[b[0]] for a, b in zip(order, order[1:]))


def run(pairs, ring, warps, groups_of, seed, batch=8):
    rng = random.Random(seed)
    nb = max(S for S, _ in pairs) + max(c for _, c in pairs) // LAG + 1
    order, _ = tickets(pairs, groups_of, nb, rng)
    members = {}
    for p, s in order:
        members.setdefault(groups_of[p], []).append((p, s))
    done, handed, buffers = {}, {}, {}  # strips finished, batches handed on, buffer -> (strip, batches)
    state = [None] * warps              # (pair, strip, next batch, claimed)
    head = 0
    while True:
        moved = False
        for w in rng.sample(range(warps), warps):
            if state[w] is None:
                if head < len(order):
                    state[w] = [*order[head], 0, False]
                    head += 1
                    moved = True
                continue
            p, s, b, claimed = state[w]
            S, cols = pairs[p]
            nbat = -(-cols // batch)
            if not claimed and s + 1 < S:  # wait for the buffer
                g = groups_of[p]
                if s >= ring and done.get((p, s - ring + 1)) is None:
                    continue
                if g >= 2 and any(t not in done for t in members.get(g - 2, [])):
                    continue
                key = (p, s % ring)
                old = buffers.get(key)
                assert old is None or (p, old[0] + 1) in done, "buffer still being read"
                buffers[key] = (s, 0)
                state[w][3] = moved = True
                continue
            if b < nbat:
                if s > 0:
                    if handed.get((p, s - 1), 0) <= b:
                        continue
                    assert buffers[p, (s - 1) % ring][0] == s - 1, "batch overwritten before it was read"
                if s + 1 < S:
                    handed[p, s] = b + 1
                state[w][2] = b + 1
            else:
                done[p, s] = True
                state[w] = None
            moved = True
        if not moved:
            break
    return len(done) == len(order) and head == len(order)


@pytest.mark.parametrize("warps", [1, 2, 5, 17])
@pytest.mark.parametrize("ring", [1, 2, 5, 100])
def test_no_interleaving_gets_stuck(warps, ring):
    for seed in range(4):
        rng = random.Random(seed)
        pairs = [(rng.randint(1, 9), rng.randint(1, 300)) for _ in range(12)]
        groups_of = sorted(rng.randint(0, 4) for _ in pairs)
        # a pair's own dependence alone never closes a cycle: with one buffer, strip s + 1 has read
        # buffer s to the end only when it is done, which needs no buffer that comes later
        assert run(pairs, max(ring, 2), warps, groups_of, seed)
