"""Routing with many picks per query (csrc/moc_route_long.cu): the picks against the oracle at the edges of its sizes, and where counting
by a threshold is hard: equal scores, chunks that repeat, rows with few candidates, scores that are not normally distributed."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU

pytestmark = pytest.mark.gpu


def ragged(heads, d, n_chunks, size, k, captions=(0,), shots=1, causal=True, window=(0, 0)):
    sizes = np.full(n_chunks, size)
    sizes[::3] += 1
    lay = W.Layout(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), (np.arange(n_chunks) * shots // n_chunks).astype(np.int32),
                   np.isin(np.arange(n_chunks), captions).astype(np.uint8))
    return W.Workload("many picks", heads, d, lay, k, *window, causal=causal)


def routed(wl, spoil=None):
    run = PU.GpuRun(wl)
    if spoil:
        spoil(run.x)
    run.forward()
    return run


def check(run):
    wl = run.wl
    orc = Oracle.from_workload(wl)
    h = run.host_inputs()
    sel = run.sel.cpu().numpy()
    PU.assert_routing(wl, orc, h["q"], orc.chunk_pool(h["k"]), sel)
    # the lists hold every pick once: the selection's pairs, as the counts in the workspace have them, are those of sel_idx
    size = np.diff(wl.layout.chunk_off).astype(np.int64)
    assert run.plan.moc_selected_pairs(run.ws) == anchor_pairs(wl) + int(size[sel[sel >= 0]].sum())


def anchor_pairs(wl):
    """Anchor pairs, by the rule."""
    lay = wl.layout
    size, text, shot, idx = np.diff(lay.chunk_off).astype(np.int64), lay.chunk_mod == 1, lay.chunk_shot, np.arange(lay.n_chunks)
    back, fwd = (lay.n_chunks if w == W.WHOLE_SHOT else w for w in (wl.win_back, wl.win_fwd))
    return wl.n_heads * sum(int(size[c]) * int(size[text | ((shot == shot[c]) & (idx >= c - back) & (idx <= c + fwd))].sum()) for c in range(lay.n_chunks))


@pytest.mark.parametrize("k", [17, 24, 25, 56, 57, 64, 120, 121, 128, 240, 241, 512])
def test_every_length_of_list(k):
    check(routed(ragged(1, 64 if k % 2 else 128, 300 if k <= 240 else 600, 5, k)))


# (survivors that are kept, by picks: 32, 64, 128, 256, 512; the first two lines lie elsewhere with more than 512 columns)
@pytest.mark.parametrize("n_chunks,k", [(300, 20), (300, 21), (300, 28), (300, 29), (300, 52), (300, 53), (300, 60), (300, 61), (600, 20), (600, 21), (600, 28), (600, 29),
                                        (600, 52), (600, 53), (600, 60), (600, 61), (600, 120), (600, 121), (600, 240), (600, 241)])
def test_every_number_of_survivors(n_chunks, k):
    check(routed(ragged(1, 128 if k % 2 else 64, n_chunks, 5, k)))


def test_one_table_of_counters():
    """So many chunks that the pick counters of a single unit fit beside the survivors; some blocks have two units and some one.  The picks against
    scores in 64 bits, the lists against those made from the selection."""
    H, C, k, d = 4, 7200, 118, 128
    lay = W.Layout(np.arange(C + 1, dtype=np.int32), np.zeros(C, np.int32), (np.arange(C) == 0).astype(np.uint8))
    run = PU.GpuRun(W.Workload("many chunks", H, d, lay, k, 0, 0)).forward()
    sel, idx = run.sel.long(), torch.arange(C, device="cuda")
    for h in range(H):
        score = run.x["q"][h].double() @ run.desc[h].double().T
        score.masked_fill_((idx[None] >= idx[:, None]) | (idx[None] == 0), -torch.inf)      # earlier chunks, but not the caption
        want = (idx - 1).clamp(0, k)
        assert torch.equal((sel[h] >= 0).sum(1), want)
        mine = torch.where(sel[h] >= 0, score.gather(1, sel[h].clamp(min=0)), torch.inf)
        kth = torch.where(want > 0, score.sort(1, descending=True).values.gather(1, (want - 1).clamp(min=0)[:, None])[:, 0], -torch.inf)
        assert bool((mine >= kth[:, None] - PU.NEAR_TIE).all())                               # none that is not among the largest
        ordered = sel[h].masked_fill(sel[h] < 0, C).sort(1).values
        assert bool(((ordered[:, 1:] > ordered[:, :-1]) | (ordered[:, 1:] == C)).all())       # none twice
        live = (sel[h, :, 1:] >= 0)
        assert bool((mine[:, :-1] >= mine[:, 1:] - PU.NEAR_TIE)[live].all())                  # best first
    O, lse, before = run.O.clone(), run.lse.clone(), run.sel.clone()
    run.plan.moc_lists_from_sel(run.sel, run.ws)
    run.attend_only()
    assert torch.equal(run.sel, before)
    assert float((run.O.float() - O.float()).abs().max()) <= 1e-2 and float((run.lse - lse).abs().max()) <= 1e-3      # the same rows, grouped into other tiles


@pytest.mark.parametrize("n_chunks,k", [(18, 33), (34, 40), (50, 40), (130, 64), (131, 64), (146, 20), (147, 20), (514, 20), (515, 30), (1026, 20), (1500, 24)])
def test_every_number_of_columns(n_chunks, k):
    check(routed(ragged(2, 64, n_chunks, 3, k, captions=(0, n_chunks // 2))))


@pytest.mark.parametrize("wl", [ragged(2, 128, 90, 17, 33, causal=False), ragged(1, 64, 1100, 3, 40, causal=False, shots=5, window=(1, 1)),
                                ragged(3, 128, 140, 20, 18, shots=7, window=(2, 0)), ragged(1, 128, 200, 9, 130, shots=4, window=(W.WHOLE_SHOT, W.WHOLE_SHOT))],
                         ids=["not causal", "not causal, 1100 chunks", "window behind", "whole shots"])
def test_candidates_that_are_not_a_prefix_or_few(wl):
    check(routed(wl))


@pytest.mark.parametrize("k,n_chunks", [(20, 200), (100, 300), (40, 1200)])
def test_equal_scores_go_to_the_earlier_chunk(k, n_chunks):
    """All scores equal: the first candidates, whatever the threshold."""
    run = routed(ragged(1, 64, n_chunks, 4, k), lambda x: x["q"].zero_())
    sel, tc = run.sel.cpu().numpy()[0], run.wl.layout.token_chunk()
    for i in range(0, len(sel), 7):
        n = min(k, max(0, int(tc[i]) - 1))                     # (chunk 0 is a caption, the row's own chunk an anchor)
        assert np.array_equal(sel[i], np.concatenate([np.arange(1, n + 1), np.full(k - n, -1)]))


def test_groups_of_equal_chunks():
    """Keys that repeat every six chunks: scores in groups of fifty equal ones, of which some are taken."""
    def repeat(x):
        off = 0
        for c, n in enumerate(np.diff(wl.layout.chunk_off)):
            x["k"][:, off:off + n] = (0.25 * base[c % 6])[:, None]
            off += n
    wl = ragged(1, 128, 301, 4, 60)
    base = torch.randint(-3, 4, (6, 1, 128), device="cuda").to(torch.bfloat16)
    run = routed(wl, repeat)
    check(run)


def test_scores_far_from_normal():
    """Scores of nine magnitudes, from a sixty-fourth to four times the usual."""
    def spread(x):
        off = np.asarray(wl.layout.chunk_off)
        for c in range(wl.n_chunks):
            x["k"][:, off[c]:off[c + 1]] *= 2.0 ** (2 - 7 * c % 9)
    wl = ragged(1, 128, 400, 4, 70)
    check(routed(wl, spread))


def blank(wl):
    """Every tenth chunk's keys zero, and scores about a negative mean: the k-th largest is often a zero, or close to it."""
    def spoil(x):
        x["q"] += 0.25
        x["k"] -= 0.25
        off = np.asarray(wl.layout.chunk_off)
        for c in range(3, wl.n_chunks, 10):
            x["k"][:, off[c]:off[c + 1]] = 0
    return spoil


BLANK = [(64, 300, 20), (128, 300, 28), (128, 400, 60), (64, 504, 118), (128, 1000, 20), (64, 1100, 52), (128, 1300, 118), (128, 700, 130)]


@pytest.mark.parametrize("d,n_chunks,k", BLANK)
def test_some_chunks_are_blank(d, n_chunks, k):
    wl = ragged(2, d, n_chunks, 4, k)
    check(routed(wl, blank(wl)))


def test_debug_build_finds_every_survivor_where_it_was_counted():
    """The build with -DMOC_DEBUG compares what a thread stores with what it counted.  (In a child process: a process loads one variant.)"""
    code = ("import sys; sys.path[:0] = %r\n"
            "import test_gpu_route_long as T\n"
            "from paper_2508_21058_b200 import lib_path\n"
            "assert lib_path().endswith('libmoc_debug.so')\n"
            "for d, n, k in T.BLANK:\n"
            "    wl = T.ragged(2, d, n, 4, k)\n"
            "    T.routed(wl, T.blank(wl))\n"
            "print('DEBUG_BUILD_OK')\n") % [PU.ROOT, os.path.join(PU.ROOT, "tests")]
    from paper_2508_21058_b200 import build as libbuild
    libbuild.build(debug=True)
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=dict(os.environ, MOC_LIBRARY="debug"), timeout=600)
    assert res.returncode == 0 and "DEBUG_BUILD_OK" in res.stdout, res.stdout[-2000:] + res.stderr[-4000:]
