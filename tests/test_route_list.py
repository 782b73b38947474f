"""The sorted list of picks of the routing kernel's few-chunk path (csrc/moc_route.cu), as a model on the CPU: scores that are not numbers are
never picked, and let nothing in that is not a candidate."""
import math
import os
import random

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_21058_b200", "csrc", "moc_route.cu")


def insert(s, j, cv, cj):
    ge = [x >= cv for x in s]
    for x in reversed(range(len(s))):
        if not ge[x]:
            first = x == 0 or ge[x - 1]
            s[x], j[x] = (cv, cj) if first else (s[x - 1], j[x - 1])


def picks(scores, candidates, k, as_none=True):
    s, j = [-math.inf] * k, [-1] * k
    for c, f in enumerate(scores):
        f = -math.inf if as_none and f != f else f
        insert(s, j, f if c in candidates else -math.inf, c)
    return j


def rows():
    rng = random.Random(3)
    for _ in range(400):
        n = rng.randint(1, 20)                               # columns; the padded ones up to 32 are no candidates
        candidates = set(range(rng.randint(0, n))) if rng.random() < 0.5 else {c for c in range(n) if rng.random() < 0.6}
        yield [rng.choice((math.nan, math.inf, -math.inf, 0.0, rng.gauss(0, 1), rng.gauss(0, 1))) for _ in range(32)], candidates, n


@pytest.mark.parametrize("k", [1, 3, 4, 8])
def test_picks_are_the_largest_numbers(k):
    for scores, candidates, _ in rows():
        real = sorted((c for c in candidates if scores[c] > -math.inf), key=lambda c: (-scores[c], c))[:k]
        assert picks(scores, candidates, k) == real + [-1] * (k - len(real))


def test_the_model_sees_what_a_score_that_is_not_a_number_lets_in():
    """Kept in the list, it is followed by columns beyond the last, which the kernel would look up in a table of that length."""
    assert any(max(picks(scores, candidates, 4, as_none=False)) >= n for scores, candidates, n in rows())


def test_the_model_is_of_this_source():
    with open(SRC) as f:
        text = f.read()
    assert "ge[x] = top.s[x] >= cv;" in text and "const bool here = x == 0 ? true : ge[x - 1];" in text
    assert "insert(((cand >> (g * 8 + c)) & 1u) ? number_or_none(f[c]) : -INFINITY, g * 8 + c);" in text
    assert 'asm("max.f32 %0, %0, 0fff800000;" : "+f"(f));' in text
