"""The ring protocol of the tensor-memory attention, on the CPU: loads land in any order, every actor runs
as soon as its parity waits let it, and no product may read a slot that does not hold its tile.
Ring positions: K of step 0, then K of step i + 1 and V of step i (csrc/attn_tc.cu)."""
import heapq
import random

import pytest


class Bar:
    """A barrier of completed phases; a wait by parity knows only whether the last one had it."""

    def __init__(self):
        self.n = 0

    def done(self, parity):
        return (self.n - 1) & 1 == parity & 1


def run(ring, steps, seed, wait_for_v):
    rnd = random.Random(seed)
    pos_k = [0] + [2 * i - 1 for i in range(1, steps)]
    pos_v = [2 * i + 2 for i in range(steps - 1)] + [2 * steps - 1]
    tile = {p: ("K", i) for i, p in enumerate(pos_k)} | {p: ("V", i) for i, p in enumerate(pos_v)}
    full, empty = [Bar() for _ in range(ring)], [Bar() for _ in range(ring)]
    s_full, s_empty, p_full, p_empty = ([Bar(), Bar()] for _ in range(4))
    held, events, now, issued = [None] * ring, [], 0, 0
    at = {"S": 0, "O": 0, "X": 0, "Xread": 0}

    def later(dt, *bars, put=None):
        heapq.heappush(events, (now + dt, rnd.random(), bars, put))

    while at["O"] < steps:
        moved = True
        while moved:
            moved = False
            use, slot = divmod(issued, ring)
            if issued < 2 * steps and (use == 0 or empty[slot].done((use & 1) ^ 1)):
                held[slot] = None
                later(rnd.choice([5, 5, 5, rnd.randint(1, 200)]), full[slot], put=(slot, tile[issued]))
                issued, moved = issued + 1, True
            i = at["S"]                                        # scores
            if i < steps:
                use, slot = divmod(pos_k[i], ring)
                if (s_empty[i & 1].done((i >> 1 & 1) ^ 1) and full[slot].done(use) and
                        (not wait_for_v or not ring & 1 or use == 0 or empty[slot].done(use - 1))):
                    if held[slot] != ("K", i):
                        return False
                    later(rnd.randint(1, 4), s_full[i & 1], empty[slot])
                    at["S"], moved = i + 1, True
            i = at["X"]                                        # softmax: reads the scores, then writes probabilities
            if i < steps and at["Xread"] == i and s_full[i & 1].done(i >> 1):
                s_empty[i & 1].n += 1
                at["Xread"], moved = i + 1, True
            if i < steps and at["Xread"] == i + 1 and (i < 2 or p_empty[i & 1].done((i >> 1 & 1) ^ 1)):
                p_full[i & 1].n += 1
                at["X"], moved = i + 1, True
            i = at["O"]                                        # outputs
            if i < steps:
                use, slot = divmod(pos_v[i], ring)
                if full[slot].done(use) and p_full[i & 1].done(i >> 1):
                    if held[slot] != ("V", i):
                        return False
                    later(rnd.randint(1, 4), p_empty[i & 1], empty[slot])
                    at["O"], moved = i + 1, True
        if at["O"] < steps:
            now, _, bars, put = heapq.heappop(events)          # (an empty heap: a deadlock, the test fails)
            if put:
                held[put[0]] = put[1]
            for b in bars:
                b.n += 1
    return True


@pytest.mark.parametrize("ring", [5, 6])
def test_products_read_their_own_tiles(ring):
    assert all(run(ring, 1 + seed % 30, seed, True) for seed in range(600))


def test_odd_ring_needs_the_wait_for_the_slot_before():
    assert not all(run(5, 1 + seed % 30, seed, False) for seed in range(600))
    assert all(run(6, 1 + seed % 30, seed, False) for seed in range(600))
