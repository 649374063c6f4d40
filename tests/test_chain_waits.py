"""CPU models of the strip chain's waits for buffers (chain_claim and chain_finish in sk_chain.cuh).

A ticket first waits until the memory it will write, and the memory it reads from, belong to its part
of the chain: until the group before the last is done (groups take the two halves of the buffers in
turn), and until the strip that last used its buffer has been read to the end.  Two models:

* Time.  Tickets are taken in order by a number of warps; a strip follows the one below it by LAG steps.
  A wait gives up when it has polled a stretch of `polls` times without any strip of the launch finishing
  meanwhile; the stretch covers one strip's sweep.  Whatever the number of groups, such a wait never gives
  up while the launch is at work, where a fixed number of polls per strip (the rule before) does.
* Memory.  Random interleavings, with buffers keyed by the memory they occupy (half, offset in the group,
  strip mod ring): no batch is overwritten before it is read, also when some claims give up, which then
  write nothing.
"""
import random

import pytest

LAG = 50          # kChainLag
WAIT_STEPS = 256  # kChainWaitSteps
LIMIT = 1 << 20   # kSpinLimit


def schedule(groups, warps, step):
    """groups: [[(strips, cols), ...], ...], every buffer of a group in its half.  step: polls that a
    sweep's step takes.  Returns the times (in polls) at which tickets finish, and the group waits as
    (first strip's place in its pair, from, to)."""
    free = [0.0] * warps
    ends, waits, group_end = [], [], []
    for g, pairs in enumerate(groups):
        tickets = sorted((-((S - s) + cols // LAG), p, s) for p, (S, cols) in enumerate(pairs) for s in range(S))
        begin, end = {}, {}
        for _, p, s in tickets:
            w = min(range(warps), key=free.__getitem__)
            start = free[w]
            ready = group_end[g - 2] if g >= 2 else 0.0
            if ready > start:
                waits.append((s, start, ready))
            b = max(start, ready, begin[p, s - 1] + LAG * step if s else 0.0)
            e = max(b + (pairs[p][1] + 31) * step, end[p, s - 1] + LAG * step if s else 0.0)
            begin[p, s], end[p, s] = b, e
            free[w] = e
            ends.append(e)
        group_end.append(max([*end.values(), group_end[-1] if g else 0.0]))
    return sorted(ends), waits


def gives_up(wait, ends, polls):
    """Whether a wait over [start, ready) sees a whole stretch of `polls` polls in which no strip finishes."""
    _, start, ready = wait
    t = start
    while t + polls < ready:
        if not any(t < e <= t + polls for e in ends):
            return True
        t += polls
    return False


SLOW = [  # groups of few pairs with refined columns near the largest allowed, slow FP64 steps (in polls)
    ([[(100, 131072)] * 2, [(100, 131072)] * 2, [(100, 131072)]], 2400, 34),
    ([[(100, 131072)], [(100, 131072)], [(100, 131072)], [(100, 131072)], [(100, 131072)]], 2400, 34),
    ([[(4, 60000), (4, 1000)], [(2, 900)], [(60, 40000)], [(3, 131072)], [(2, 32)]], 64, 200),
    ([[(30, 5000)]] * 7, 1000, 20),
]


@pytest.mark.parametrize("groups,warps,step", SLOW)
def test_a_wait_for_a_group_lasts_while_strips_finish(groups, warps, step):
    ends, waits = schedule(groups, warps, step)
    assert waits
    cols = max(c for pairs in groups for _, c in pairs)
    polls = LIMIT * (1 + (cols + 31) // WAIT_STEPS)
    assert not any(gives_up(w, ends, polls) for w in waits)
    # the bound has room: a strip's sweep is a small part of a stretch
    assert 4 * (cols + 31) * step <= polls


def test_a_fixed_number_of_polls_runs_out_on_a_slow_group():
    """The rule before: (strip + 1) x the limit, for the whole group.  Five pairs of 3200 x 131072 cells, two
    to a half of the buffers: the fifth pair's first strip waits for the first two pairs."""
    ends, waits = schedule(*SLOW[0])
    assert any(to - frm > LIMIT * (s + 1) for s, frm, to in waits)


def test_progress_alone_runs_out_on_a_long_strip():
    """Progress is counted in finished strips, so a stretch has to cover one strip's sweep."""
    groups, warps, step = SLOW[1]
    ends, waits = schedule(groups, warps, step)
    assert any(gives_up(w, ends, LIMIT) for w in waits)


def test_a_launch_that_stands_still_is_given_up():
    """No strip finishes any more: the wait ends after one stretch."""
    assert gives_up((0, 0.0, float(1 << 40)), [10.0, 500.0], 1000)


def interleave(groups, ring, warps, seed, group_wait=True, ring_wait=True, give_up=0.0, writes_on=False, batch=8):
    """Random interleaving; returns whether every ticket ended.  group_wait / ring_wait: leave a wait out (a
    planted mistake).  give_up: probability that a claim that has to wait gives up; it then writes nothing
    (writes_on: it does, a planted mistake), and the strips after it give up their reads."""
    rng = random.Random(seed)
    order, at = [], {}
    for g, pairs in enumerate(groups):
        off = 0
        keyed = []
        for p, (S, cols) in enumerate(pairs):
            for s in range(S):
                k = s % min(ring, S - 1) if S > 1 else 0
                at[g, p, s] = (g & 1, off + k)
                keyed.append((-((S - s) + cols // LAG), rng.random(), (g, p, s)))
            off += min(S - 1, ring)
        order += [t for _, _, t in sorted(keyed)]
    left = {g: sum(S for S, _ in pairs) for g, pairs in enumerate(groups)}
    done, handed, memory, failed = set(), {}, {}, set()  # memory: place -> the ticket whose columns it holds
    state = [None] * warps
    head = 0
    while True:
        moved = False
        for w in rng.sample(range(warps), warps):
            if state[w] is None:
                if head < len(order):
                    state[w] = [order[head], 0, "claim", False]
                    head += 1
                    moved = True
                continue
            (g, p, s), b, phase, mute = state[w]
            S, cols = groups[g][p]
            nbat = -(-cols // batch)
            last = s + 1 == S
            if phase == "claim":
                v = s - 1 if last else s  # whose buffer the ring wait is for
                blocked = group_wait and g >= 2 and left[g - 2] > 0
                blocked = blocked or (ring_wait and v >= ring and (g, p, v - ring + 1) not in done)
                if blocked and rng.random() >= give_up:
                    continue
                if blocked:
                    failed.add((g, p))
                    mute = not writes_on
                if not last and not mute:
                    old = memory.get(at[g, p, s])
                    if old is not None and old[:2] not in failed:
                        assert (old[0], old[1], old[2] + 1) in done, "buffer still being read"
                    memory[at[g, p, s]] = (g, p, s)
                state[w] = [(g, p, s), 0, "sweep", mute]
                moved = True
                continue
            if b < nbat:
                if s > 0 and (g, p) not in failed:
                    if handed.get((g, p, s - 1), 0) <= b:
                        continue
                    assert memory[at[g, p, s - 1]] == (g, p, s - 1), "batch overwritten before it was read"
                if not last and not mute:
                    handed[g, p, s] = b + 1
                state[w][1] = b + 1
            else:
                done.add((g, p, s))
                left[g] -= 1
                state[w] = None
            moved = True
        if not moved and not (give_up and any(t and t[2] == "claim" for t in state)):
            break
    return head == len(order) and len(done) == len(order)


def some_groups(rng):
    return [[(rng.randint(1, 7), rng.randint(1, 120)) for _ in range(rng.randint(1, 3))] for _ in range(5)]


@pytest.mark.parametrize("warps", [1, 3, 24])
@pytest.mark.parametrize("ring", [2, 3, 100])
def test_memory_is_not_overwritten(warps, ring):
    for seed in range(30):
        assert interleave(some_groups(random.Random(seed)), ring, warps, seed)


def test_two_strip_pairs_use_one_buffer():
    for seed in range(20):
        assert interleave([[(2, 100), (2, 40)], [(2, 60)], [(2, 9)], [(1, 5)], [(2, 77)]], 1, 6, seed)


@pytest.mark.parametrize("warps", [3, 24])
def test_a_claim_that_gives_up_writes_nothing(warps):
    for seed in range(30):
        assert interleave(some_groups(random.Random(seed)), 2, warps, seed, give_up=0.02)


@pytest.mark.parametrize("mistake", [dict(group_wait=False), dict(ring_wait=False), dict(give_up=0.3, writes_on=True)])
def test_the_memory_model_sees_a_missing_wait(mistake):
    caught = 0
    for seed in range(40):
        try:
            interleave(some_groups(random.Random(seed)), 2, 24, seed, **mistake)
        except AssertionError:
            caught += 1
    assert caught > 0
