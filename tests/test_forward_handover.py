"""The hand-overs of an item between the warps of the forward attention kernel (csrc/moc_attend_tc.cu), as a model of its
mbarriers that is run under many schedules on the CPU: no wait may miss its phase.  One softmax agent stands for a group of
128 threads and one key tile for an item; the barriers that lie within an item are left out where others imply them."""
import os
import random
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_21058_b200", "csrc", "moc_attend_tc.cu")
AGENTS = ("scheduler", "loader", "bookkeeping", "issuer 0", "issuer 1", "softmax 0", "softmax 1", 0, 1)      # 0, 1: the issuers' queues


class Barrier:
    def __init__(self, need=1):
        self.need, self.got, self.phase = need, 0, 0

    def arrive(self):
        self.got += 1
        if self.got == self.need:
            self.got, self.phase = 0, self.phase + 1

    def done(self, parity):                              # as the hardware's wait by parity: the phase before the current one
        return (self.phase & 1) != parity


def run(tiles, seed, slow, rows_done=4, claim="after the tile is there"):
    """One schedule of items with the given numbers of query tiles (1 or 2), `slow` held back; each item is claimed late, that is
    when the last S of the one before has been issued.  Returns whether all came to their end, and whether an item was
    claimed too early."""
    rng, n_items = random.Random(seed), len(tiles)
    q_full, q_empty = [Barrier() for _ in range(6)], [Barrier() for _ in range(3)]
    item_full, item_empty = [Barrier() for _ in range(2)], [Barrier(6) for _ in range(2)]
    s_full, p_full, o_full, turn = ([Barrier(), Barrier()] for _ in range(4))
    done = [Barrier() for _ in range(2 * rows_done)]
    slot, pipe, released, early = [0, 0], [[], []], set(), []

    def items():                                         # what every reader of the item ring does first
        n = 0
        while True:
            yield n, lambda: item_full[n & 1].done(n >> 1 & 1)
            n += 1

    def scheduler():
        n_q, last_g, phase = 0, 0, [0] * 6
        for n in range(n_items + 1):
            if n >= 2:
                yield lambda: item_empty[n & 1].done(n - 2 >> 1 & 1)
            if n:
                b, use = (n_q - 1) % 3, (n_q - 1) // 3
                if claim == "after the tile is there":
                    yield lambda: q_full[3 * last_g + b].done(phase[3 * last_g + b] ^ 1)
                elif claim == "after the use before" and use:
                    yield lambda: q_empty[b].done(use - 1 & 1)
                yield lambda: q_empty[b].done(use & 1)
                early.append(n_q - 1 not in released)
            slot[n & 1] = tiles[n] if n < n_items else 0
            item_full[n & 1].arrive()
            last_g = slot[n & 1] - 1
            for g in range(slot[n & 1]):
                phase[3 * g + n_q % 3] ^= 1
                n_q += 1
            yield None

    def loader():
        n_q = 0
        for n, published in items():
            yield published
            qt = slot[n & 1]
            item_empty[n & 1].arrive()
            if not qt:
                return
            for g in range(qt):
                yield lambda: q_empty[n_q % 3].done(n_q // 3 & 1 ^ 1)
                q_full[3 * g + n_q % 3].arrive()
                n_q += 1
                yield None

    def issuer(g):
        n_q, mine, phase = 0, 0, [0, 0, 0]
        for n, published in items():
            yield published
            qt = slot[n & 1]
            item_empty[n & 1].arrive()
            if not qt:
                return
            tile, n_q = n_q + g, n_q + qt
            b = tile % 3
            if g >= qt:
                continue
            yield lambda: q_full[3 * g + b].done(phase[b])
            phase[b] ^= 1
            pipe[g] += [s_full[g].arrive, lambda b=b, tile=tile: (released.add(tile), q_empty[b].arrive())]
            yield lambda: p_full[g].done(mine & 1)
            pipe[g].append(o_full[g].arrive)
            mine += 1

    def softmax(g):
        mine, turns = 0, 0
        for n, published in items():
            yield published
            qt = slot[n & 1]
            item_empty[n & 1].arrive()
            if not qt:
                return
            if g >= qt:
                continue
            yield lambda: s_full[g].done(mine & 1)
            if qt == 2:
                if g == 1 or turns:
                    yield lambda: turn[g ^ 1].done((turns if g else turns - 1) & 1)
                turn[g].arrive()
                turns += 1
            p_full[g].arrive()
            yield lambda: o_full[g].done(mine & 1)
            mine += 1
            done[2 * (n % rows_done) + g].arrive()
            yield None

    def bookkeeping():
        before, phase = 0, [0] * (2 * rows_done)
        for n, published in items():
            yield published
            for g in range(before):
                b = 2 * ((n - 1) % rows_done) + g
                yield lambda: done[b].done(phase[b])
                phase[b] ^= 1
            yield None
            before = slot[n & 1]
            item_empty[n & 1].arrive()
            yield None
            if not before:
                return

    agents = dict(zip(AGENTS, (scheduler(), loader(), bookkeeping(), issuer(0), issuer(1), softmax(0), softmax(1))))
    waits, left = dict.fromkeys(agents), list(agents)
    while left or any(pipe):
        ready = [a for a in left if waits[a] is None or waits[a]()] + [g for g in (0, 1) if pipe[g]]
        if not ready:
            return False, any(early)                     # a wait that nothing will end
        who = rng.choice([a for a in ready if a != slow] or ready) if rng.random() < 0.97 else rng.choice(ready)
        if who in (0, 1):
            pipe[who].pop(0)()
            continue
        try:
            waits[who] = next(agents[who])
        except StopIteration:
            left.remove(who)
    return True, any(early)


def _schedules(**kw):
    for slow in (None, *AGENTS):
        for seed in range(120):
            rng = random.Random(seed)
            yield run([rng.choice((1, 2, 2)) for _ in range(2 + seed % 12)], seed, slow, **kw)


def test_the_model_is_of_this_source():
    with open(SRC) as f:
        text = f.read()
    assert re.findall(r"bar\(ROWS_DONE \+ (.+)\)\);", text) == ["2 * ((n_item - 1) & 3) + g"]
    assert "const int b = 2 * ((n_item - 2) & 3) + g;" in text
    late = text[text.index("total <= 2 * (int)gridDim.x"):]
    assert late.index("if (LOADERS) ok = mbar_wait(bar(Q_FULL + qf)") < late.index("mbar_wait(bar(Q_EMPTY + qb)")


def test_no_warp_waits_for_good_and_none_goes_on_too_early():
    assert all(ended and not early for ended, early in list(_schedules()))


def test_the_model_sees_a_barrier_per_slot_miss_a_phase():
    """Two sets of ROWS_DONE, as many as item slots: the bookkeeping lane, held back, misses a phase."""
    assert not all(ended for ended, _ in list(_schedules(rows_done=2)))


def test_the_model_sees_a_late_claim_that_is_not():
    """A buffer's release taken for the next one's (Q_EMPTY waited for alone), or missed (the one before waited for first)."""
    assert any(early for _, early in list(_schedules(claim="at once")))
    assert not all(ended for ended, _ in list(_schedules(claim="after the use before")))
