"""The forward attention kernel's ring of items (csrc/moc_attend_tc.cu): slots, counts of stored rows and what a phase of the queue
waits for, as a model of its mbarriers that is run under many schedules on the CPU.  No wait by parity may miss its phase."""
import random
import re

from test_forward_handover import SRC, Barrier

AGENTS = ("scheduler", "loader", "bookkeeping", "softmax 0", "softmax 1")


def run(items, seed, slow, slots=3, rows_done=4, skip_waits=True):
    """One schedule of items (query tiles, phase), `slow` held back.  A phase's first item waits for something (DEPEND).  Returns
    whether every agent came to its end and nobody went through a DEPEND that was not there."""
    rng, n_items = random.Random(seed), len(items)
    full, empty = [Barrier() for _ in range(slots)], [Barrier(4) for _ in range(slots)]
    done, depend = [Barrier() for _ in range(2 * rows_done)], Barrier()
    slot, released, wrong = [None] * slots, [0], []

    def published():
        for n in range(n_items + 1):
            yield n, (lambda n=n: full[n % slots].done(n // slots & 1))

    def scheduler():
        for n in range(n_items + 1):
            if n >= slots:
                yield lambda: empty[n % slots].done(n // slots - 1 & 1)
            slot[n % slots] = items[n] if n < n_items else None
            full[n % slots].arrive()
            yield None

    def loader():
        for n, ready in published():
            yield ready
            last = slot[n % slots] is None
            empty[n % slots].arrive()
            if last:
                return

    def softmax(g):
        seen, deps = None, 0
        for n, ready in published():
            yield ready
            item = slot[n % slots]
            empty[n % slots].arrive()
            if item is None:
                return
            tiles, phase = item
            first, seen = phase != seen, phase
            if first:
                deps += 1
            if g >= tiles:
                if first and skip_waits:
                    yield lambda: depend.done(deps - 1 & 1)
                    wrong.append(released[0] < deps)
                    done[2 * (n % rows_done) + 1].arrive()
                continue
            yield None                                       # its tiles
            if first:
                yield lambda: depend.done(deps - 1 & 1)
                wrong.append(released[0] < deps)
            done[2 * (n % rows_done) + g].arrive()
            yield None

    def bookkeeping():
        wait_for, phase, seen = 0, [0] * (2 * rows_done), None
        for n, ready in published():
            yield ready
            item = slot[n % slots]
            for g in range(wait_for):
                b = 2 * ((n - 1) % rows_done) + g
                yield lambda: done[b].done(phase[b])
                phase[b] ^= 1
            empty[n % slots].arrive()
            yield None                                       # its fence and count, as long as they take
            if item is None:
                return
            first, seen = item[1] != seen, item[1]
            if first:
                released[0] += 1
                depend.arrive()
            wait_for = 2 if item[0] == 2 or (first and skip_waits) else 1

    agents = dict(zip(AGENTS, (scheduler(), loader(), bookkeeping(), softmax(0), softmax(1))))
    waits, left = dict.fromkeys(agents), list(agents)
    while left:
        able = [a for a in left if waits[a] is None or waits[a]()]
        if not able:
            return False                                     # a wait that nothing will end
        who = rng.choice([a for a in able if a != slow] or able) if rng.random() < 0.97 else rng.choice(able)
        try:
            waits[who] = next(agents[who])
        except StopIteration:
            left.remove(who)
    return not any(wrong)


def _schedules(**kw):
    for slow in (None, *AGENTS):
        for seed in range(150):
            rng, phase, items = random.Random(seed), 0, []
            for _ in range(3 + seed % 20):
                phase += rng.random() < 0.3
                items.append((rng.choice((1, 1, 2)), phase))
            yield run(items, seed, slow, **kw)


def test_the_model_is_of_this_source():
    with open(SRC) as f:
        text = f.read()
    assert re.findall(r"constexpr int kItemSlots = (\d);", text) == ["3"]
    assert "pend_tiles = it_.rows > 128 || dep_anchor || dep_routed ? 2 : 1;" in text
    assert "for (int t = 0; t < 8; ++t) mbar_init(bar(ROWS_DONE + t), 128);" in text


def test_no_warp_misses_a_phase():
    assert all(_schedules())


def test_the_model_sees_a_ring_that_is_too_long():
    """A slot more than the ROWS_DONE allow for: the bookkeeping lane, held back, misses a phase."""
    assert not all(_schedules(slots=4))


def test_the_model_sees_a_group_that_does_not_wait():
    """A group without a tile in a phase's first item that leaves its DEPEND out takes the next one's for its own, or misses one."""
    assert not all(_schedules(skip_waits=False))
