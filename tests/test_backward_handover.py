"""The hand-overs between the warps of the dK/dV kernel (csrc/moc_attend_bwd_tc.cu), as a model of its mbarriers that is run
under many schedules on the CPU: whoever reads a stage of a ring or a tensor-memory tile must find the tile it means.  The
barrier operations of the two issuing warps are read off the source, so that the model and the kernel cannot part."""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_21058_b200", "csrc", "moc_attend_bwd_tc.cu")
Y1, Y2 = 3, 2                                            # stages of the Q and dO rings
# what the loop of each issuing warp does per tile, in order: (wait | commit | arrive, barrier, parity) and its MMA groups;
# "+": only where there is a next tile
SIDE1 = ["wait Y2_FULL + (j & 1), (j >> 1) & 1", "wait P_HALF, j & 1", "acc2 0", "+wait Y1_FULL + s3n, ph3n", "wait P_DONE, j & 1", "acc2 1",
         "+t1", "+commit T1_FULL + ((j + 1) & 1)", "commit Y2_EMPTY + (j & 1)", "+arrive T1_ISSUED + (j & 1)"]
SIDE2 = ["+wait T1_ISSUED + (j & 1), (j >> 1) & 1", "wait DS_DONE + (j & 1), (j >> 1) & 1", "acc1", "commit Y1_EMPTY + s3",
         "+wait Y2_FULL + (jn & 1), (jn >> 1) & 1", "+t2", "+commit T2_FULL + (jn & 1)", "+commit Y2_EMPTY + (jn & 1)"]


def source_ops(text):
    """The operations of an issuer's loop over the tiles, in the form of the lists above."""
    ops = []
    pat = r"\bwait\((.+), BW_\w+\)|tc_commit_elect\(bar\((.+)\)\);|mbar_arrive\(bar\((.+)\)\);|\b(acc2)\(j, (\d)\)|\b(acc1|t1|t2)\("
    for line in text[text.index("for (int j = 0;"):].splitlines():
        for m in re.finditer(pat, line.split("//")[0]):
            w, c, a, acc2, half, mma = m.groups()
            ops.append(f"wait {w}" if w else f"commit {c}" if c else f"arrive {a}" if a else f"{acc2} {half}" if acc2 else mma)
    return ops


class Barrier:
    def __init__(self, need):
        self.need, self.got, self.phase = need, 0, 0

    def arrive(self):
        self.got += 1
        if self.got == self.need:
            self.got, self.phase = 0, self.phase + 1

    def done(self, parity):                              # as the hardware's wait by parity: the phase before the current one
        return (self.phase & 1) != parity


class WrongTile(Exception):
    pass


def run(n, side1, side2, seed, slow):
    """One schedule of n tiles; `slow` is held back.  Raises WrongTile; returns whether every warp came to its end."""
    rng = random.Random(seed)
    bars = {f"{b}{i}": Barrier(2 if b == "Y2_EMPTY" else 1) for b in ("Y1_FULL", "Y1_EMPTY", "Y2_FULL", "Y2_EMPTY", "T1_FULL", "T2_FULL", "P_HALF",
                                                                     "P_DONE", "DS_DONE", "T1_ISSUED") for i in range(3)}
    mem, pipe = {}, {"w12": [], "w13": []}               # contents; MMAs and commits still in each issuer's queue

    def bar(expr, env):
        name = re.match(r"\w+", expr).group()
        return bars[f"{name}{eval(expr.replace(name, '0', 1), {}, env)}"]

    def want(where, what):
        if mem.get(where) != what:
            raise WrongTile(f"{where} holds {mem.get(where)}, not {what}")

    def mma(reads, writes):
        def go():
            for r in reads:
                want(*r)
            for where, what in writes:
                mem[where] = what
        return go

    def groups(op, j):
        jn = j + 1
        return {"t1": lambda: mma([(f"Y1_{jn % Y1}", jn)], [("T1", jn)]), "t2": lambda: mma([(f"Y2_{jn % Y2}", jn)], [("T2", jn)]),
                "acc1": lambda: mma([(f"Y1_{j % Y1}", j), ("T2", ("dS", j))], []),
                "acc2 0": lambda: mma([(f"Y2_{j % Y2}", j), ("T1 first half", j)], []),
                "acc2 1": lambda: mma([(f"Y2_{j % Y2}", j), ("T1", ("P", j))], [])}[op]()

    def issuer(who, ops, first):
        yield from first(pipe[who].append)
        for j in range(n):
            env = dict(j=j, jn=j + 1, s3=j % Y1, s3n=(j + 1) % Y1, ph3n=(j + 1) // Y1 & 1)
            for op in ops:
                if op[0] == "+" and j + 1 == n:
                    continue
                op = op.lstrip("+")
                kind, _, rest = op.partition(" ")
                if kind == "wait":
                    b, parity = rest.rsplit(", ", 1)
                    b, parity = bar(b, env), eval(parity, {}, env)
                    yield lambda: b.done(parity)
                elif kind == "commit":
                    pipe[who].append(bar(rest, env).arrive)
                elif kind == "arrive":
                    bar(rest, env).arrive()
                    yield None
                else:
                    pipe[who].append(groups(op, j))

    def first1(put):
        yield lambda: bars["Y1_FULL0"].done(0)
        put(mma([("Y1_0", 0)], [("T1", 0)]))
        put(bars["T1_FULL0"].arrive)

    def first2(put):
        yield lambda: bars["Y2_FULL0"].done(0)
        put(mma([("Y2_0", 0)], [("T2", 0)]))
        put(bars["T2_FULL0"].arrive)
        put(bars["Y2_EMPTY0"].arrive)

    def producer(ring, stages):
        for j in range(n):
            st, ph = j % stages, j // stages & 1
            yield lambda: bars[f"{ring}_EMPTY{st}"].done(ph ^ 1)
            mem[f"{ring}_{st}"] = j
            yield None
            if ring == "Y1":
                if j >= 2:
                    yield lambda: bars[f"DS_DONE{j & 1}"].done((j - 2) >> 1 & 1)
                mem[f"ld_{j & 1}"] = j
            bars[f"{ring}_FULL{st}"].arrive()

    def lanes():
        for j in range(n):
            yield lambda: bars[f"T1_FULL{j & 1}"].done(j >> 1 & 1)
            yield lambda: bars[f"Y1_FULL{j % Y1}"].done(j // Y1 & 1)
            want("T1", j)
            want(f"ld_{j & 1}", j)
            mem["T1 first half"] = j
            bars["P_HALF0"].arrive()
            yield None
            mem["T1"] = ("P", j)
            bars["P_DONE0"].arrive()
            yield lambda: bars[f"T2_FULL{j & 1}"].done(j >> 1 & 1)
            want("T2", j)
            want(f"ld_{j & 1}", j)
            mem["T2"] = ("dS", j)
            bars[f"DS_DONE{j & 1}"].arrive()

    agents = {"Q": producer("Y1", Y1), "dO": producer("Y2", Y2), "lanes": lanes(), "w12": issuer("w12", side1, first1), "w13": issuer("w13", side2, first2)}
    waits = {a: None for a in agents}
    left = set(agents)
    while left or any(pipe.values()):
        ready = [a for a in left if waits[a] is None or waits[a]()] + [("pipe", w) for w in pipe if pipe[w]]
        if not ready:
            return False                                 # a wait that nothing will end
        fast = [a for a in ready if a != slow] or ready
        who = rng.choice(fast if rng.random() < 0.97 else ready)
        if isinstance(who, tuple):
            pipe[who[1]].pop(0)()
            continue
        try:
            waits[who] = next(agents[who])
        except StopIteration:
            left.discard(who)
    return True


def _schedules(side1, side2):
    for slow in (None, "Q", "dO", "lanes", "w12", "w13", ("pipe", "w12"), ("pipe", "w13")):
        for seed in range(60):
            yield run(1 + seed % 9, side1, side2, seed, slow)


def test_the_model_is_of_this_source():
    with open(SRC) as f:
        side1, side2 = f.read().split("if (side1) {")[1].split("} else {")[:2]
    assert source_ops(side1) == [op.lstrip("+") for op in SIDE1]
    assert source_ops(side2) == [op.lstrip("+") for op in SIDE2] + ["commit ACC_FULL"]


def test_every_reader_finds_its_tile_and_every_warp_ends():
    assert all(list(_schedules(SIDE1, SIDE2)))


@pytest.mark.parametrize("missing", ["wait Y2_FULL + (j & 1), (j >> 1) & 1", "wait P_DONE, j & 1", "+wait Y1_FULL + s3n, ph3n"])
def test_the_model_sees_a_missing_wait(missing):
    with pytest.raises(WrongTile):
        list(_schedules([op for op in SIDE1 if op != missing], SIDE2))


def test_the_model_sees_a_barrier_that_gets_two_phases_ahead():
    """One barrier in the place of the pair: the dS side, held back, misses a phase and waits for good."""
    one = [[op.replace("T1_ISSUED + (j & 1), (j >> 1) & 1", "T1_ISSUED, j & 1").replace("T1_ISSUED + (j & 1)", "T1_ISSUED") for op in ops]
           for ops in (SIDE1, SIDE2)]
    assert not all(list(_schedules(*one)))


def shared_tile_epilogue(seed, s_last, initialised):
    """The end of a block that shares its key tile (two barriers of the lane warps, the count of the blocks that have left their sums in
    between), in which waits for a barrier that is not complete may run out.  Whether a warp stored although the block has not
    counted itself, and so does not know that it is the last."""
    rng, bars, state = random.Random(seed), (Barrier(8), Barrier(8)), {"last": 0 if initialised else s_last, "counted": False}
    stored = []

    def warp(w):
        ok = True
        bars[0].arrive()
        yield 0, lambda: bars[0].done(0)
        ok = ok and bars[0].done(0)
        if w == 0 and ok:
            state.update(last=1, counted=True)               # this block is the last one
        bars[1].arrive()
        if ok:
            yield 1, lambda: bars[1].done(0)
            ok = bars[1].done(0)
        if ok and state["last"]:
            stored.append(state["counted"])

    agents = {w: warp(w) for w in range(8)}
    waits, slow = dict.fromkeys(agents), rng.randrange(8)
    while agents:
        able = [w for w in agents if waits[w] is None or waits[w][1]()]
        late = [w for w in agents if w not in able and rng.random() < 0.2]      # ... and these run out
        who = rng.choice([w for w in able + late if w != slow] or able or list(agents))
        try:
            waits[who] = next(agents[who])
        except StopIteration:
            del agents[who]
    return not all(stored)


def test_a_block_that_gives_up_on_a_shared_tile_stores_nothing():
    with open(SRC) as f:
        text = f.read()
    before = text[:text.index("__syncthreads();")]
    assert any(shared_tile_epilogue(seed, 1, False) for seed in range(500))      # the model sees what an unset flag does
    assert not any(shared_tile_epilogue(seed, 1, True) for seed in range(500))
    assert re.search(r"\bs_last = 0;", before)                                   # and the kernel sets it before the barriers are used
