"""The search for a threshold of the routing kernel for many picks (csrc/moc_route_long.cu), as a model of one row on the CPU: what is counted
is what is stored, and the picks are the largest scores, whatever the mixture of zeros, subnormal numbers and ordinary scores."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_21058_b200", "csrc", "moc_route_long.cu")
F = np.float32
TINY, MAX, SEGMENT = np.finfo(F).tiny, np.finfo(F).max, 512


def flushed(x):
    return np.where(np.abs(x) < TINY, F(0), x).astype(F)


def bits(x):
    return int(np.asarray(x, F).view(np.uint32))


def ordered(x):
    return ~bits(x) & 0xffffffff if bits(x) >> 31 else bits(x) | 0x80000000


def from_ordered(u):
    return np.array(u ^ 0x80000000 if u >> 31 else ~u & 0xffffffff, np.uint32).view(F)[()]


def normal_above(p):
    with np.errstate(all="ignore"):                       # (not a number where p is 0 or 1)
        t = np.sqrt(F(-2) * np.log(F(min(p, F(1) - p))))
        z = t - (F(2.515517) + t * (F(0.802853) + t * F(0.010328))) / (F(1) + t * (F(1.432788) + t * (F(0.189269) + t * F(0.001308))))
    return F(z) if p <= 0.5 else F(-z)


def taken(f, col, thr, before):
    f, thr = flushed(f), flushed(thr)
    return (f > thr) | ((f == thr) & (col < before))


def search(scores, k, cap, flush_in_store=True):
    """Picks of a row whose candidates are all its columns, and whether every count of survivors was the number stored."""
    surv, col, same = np.empty(0, F), np.empty(0, int), True
    for seg in range(0, len(scores), SEGMENT):
        v, j = scores[seg:seg + SEGMENT], np.arange(seg, min(len(scores), seg + SEGMENT))
        so_far = scores[:seg + SEGMENT]
        n = len(so_far)
        inv = F(1) / F(n)
        mean = F(so_far.sum(dtype=F) * inv)
        sd = np.sqrt(max(F((so_far * so_far).sum(dtype=F) * inv - mean * mean), F(0)))
        found, thr = n <= cap, F(-MAX)
        low, high, z_low, z_high = ordered(F(-MAX)), ordered(F(np.inf)) + 1, F(np.nan), F(np.nan)
        before, b_low, b_high = 1 << 31, 0, 0

        def in_between(guess, thr):
            key = ordered(thr)
            if not guess or not low < key < high:
                key = low + (high - low >> 1)
            return from_ordered(key)

        if not found:
            z = normal_above(F(0.5) * F(k + cap) * inv)
            thr = in_between(True, F(mean + z * sd))
        for it in range(400):
            total = int(taken(v, j, thr, before).sum() + taken(surv, col, thr, before).sum())
            found = found or k <= total <= cap
            if found:
                break
            if before == 1 << 31:
                z_thr = normal_above(max(F(total), F(0.5)) * inv)
                if total > cap:
                    low, z_low = ordered(thr), z_thr
                else:
                    high, z_high = ordered(thr), z_thr
                if high - low <= 1:
                    thr, b_high = from_ordered(low), 1 << 16
                else:
                    t_low, t_high = from_ordered(low), from_ordered(high)
                    with np.errstate(all="ignore"):
                        guess = t_low + (t_high - t_low) * ((z - z_low) / (z_high - z_low)) if z_low < z_high else thr + sd * (z - z_thr)
                    thr = in_between(it & 3 != 3, F(guess))
            elif total > cap:
                b_high = before
            else:
                b_low = before
            if b_high:
                before = b_low + (b_high - b_low >> 1)
            if b_high and b_high - b_low <= 1:
                before, found = b_high, True
        else:
            raise AssertionError("the search does not end")
        total = int(taken(v, j, thr, before).sum() + taken(surv, col, thr, before).sum())
        keep = taken(surv, col, thr, before)
        new = taken(v, j, thr, before)
        if not flush_in_store and before == 1 << 31:      # (rows with a bound on the column are stored as they are counted)
            new = v >= thr
        surv, col = np.concatenate([surv[keep], v[new]]), np.concatenate([col[keep], j[new]])
        same = same and len(surv) == total
    order = np.lexsort((col, -flushed(surv).astype(np.float64)))
    return col[order][:k], same


def rows(seed, n_rows, n, zeros, mean, kind):
    """Normal scores, some of which are zero, or subnormal."""
    rng = np.random.RandomState(seed)
    for _ in range(n_rows):
        x = (rng.randn(n) + mean).astype(F)
        at = rng.permutation(n)[:zeros]
        x[at] = 0
        if kind != "zeros":
            some = at[::2] if kind == "mixed" else at
            x[some] = (rng.uniform(-1, 1, len(some)) * TINY).astype(F)
        if kind == "small":                               # all scores around the smallest normal number
            x = (x * F(4) * TINY).astype(F)
        yield x


MIXTURES = [(300, 20, 32, 12), (300, 28, 32, 1), (400, 60, 64, 30), (504, 40, 64, 40), (504, 118, 128, 100), (330, 17, 32, 20), (309, 34, 64, 32),
            (1008, 20, 32, 12), (1008, 52, 64, 100), (1200, 118, 128, 60), (90, 60, 64, 40)]


@pytest.mark.parametrize("n,k,cap,zeros", MIXTURES)
@pytest.mark.parametrize("kind", ["zeros", "mixed", "subnormal", "small"])
def test_survivors_are_those_counted_and_picks_the_largest(n, k, cap, zeros, kind):
    for seed, mean in enumerate((-1.8, -1.5, -1.3, -0.5, 0.0, 1.0)):
        for x in rows(seed, 12, n, zeros, mean, kind):
            picks, same = search(x, k, cap)
            assert same
            assert np.array_equal(picks, np.lexsort((np.arange(n), -flushed(x).astype(np.float64)))[:k])


def test_the_model_is_of_this_source():
    with open(SRC) as f:
        text = f.read()
    assert text.count("setp.ge.ftz.f32") == 1 and not re.search(r"setp\.\w+(\.and|\.or)?\.f32", text)             # the rule alone compares
    search_code = text[text.index("// A threshold that at least k"):text.index("// a warp per row, two rows at a time")]
    assert len(re.findall(r"reaches\(", search_code)) == 7 and not re.findall(r"([<>]|[<>=]=) thr\b|\bthr ([<>]|==)", search_code)
    assert "return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);" in text and "(u & 0x80000000u) ? u ^ 0x80000000u : ~u" in text
    assert "(uint64_t)sort_key(sc_at(r0 + 4 * b, x)) << 32" in text


def test_the_model_sees_a_store_that_tells_subnormals_from_zero():
    """Some thresholds are subnormal, and so are some scores: the counts are not what is stored."""
    assert not all(search(x, 60, 64, False)[1] for x in rows(7, 300, 400, 30, -1.3, "zeros"))
    assert not all(search(x, 34, 64, False)[1] for x in rows(8, 100, 309, 32, -1.5, "small"))
