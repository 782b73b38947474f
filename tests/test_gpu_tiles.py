"""The attention and routing kernels at the edges of their tiles, lists and variants, against the CPU oracle, with the
tolerances of the other parity tests; and a workspace used again gives the same bits."""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU

pytestmark = pytest.mark.gpu

# heads, head_dim, (shots, caption, frames, frame length), k
SHAPES = {
    "whole tiles only": (5, 128, (3, 128, 6, 128), 4),                 # one key tile a chunk; every dK/dV query tile from consecutive rows
    "four key tiles a chunk": (2, 128, (2, 16, 4, 512), 2),            # the last size with four query-loading warps
    "four key tiles and one key": (2, 128, (2, 16, 4, 513), 2),        # the first with one
    "two key tiles a chunk": (2, 128, (2, 16, 6, 256), 2),
    "two key tiles and one key": (2, 128, (2, 16, 8, 257), 6),         # three key tiles, the last with one key; whole batches of the merge
    "three key tiles, 7 picks": (2, 128, (2, 16, 8, 384), 7),          # a last merge batch with one slot
    "four key tiles, 8 picks": (1, 128, (2, 16, 8, 512), 8),           # ... with two
    "four key tiles, 9 picks": (1, 128, (2, 16, 8, 512), 9),
    "one row past a tile": (7, 128, (2, 1, 11, 129), 9),               # items of 256 rows and of a few; a merge of 8 + 1 picks
    "one row short of two tiles": (2, 64, (2, 31, 9, 255), 8),         # a full merge batch
    "17 picks": (3, 64, (2, 1, 13, 65), 17),                           # the shortest sorted list, 26 columns
    "32 picks of 33 columns and more": (2, 128, (3, 8, 15, 33), 32),   # a full list, and one column in the second block
    "33 picks": (2, 64, (2, 8, 24, 33), 33),                           # the longer list
    "fewer candidates than picks": (2, 128, (1, 8, 20, 40), 24),
    "no picks": (3, 128, (2, 130, 3, 129), 0),                         # anchor items alone
}


@pytest.mark.parametrize("shape", SHAPES)
def test_tile_and_list_edges(shape):
    heads, d, lay, k = SHAPES[shape]
    wl = W.Workload("edges", heads, d, W.make_layout(*lay), k, 1, 1)
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
    x, orc = run.host_inputs(), Oracle.from_workload(wl)
    sel = run.sel.cpu().numpy()
    if k:
        PU.assert_routing(wl, orc, x["q"], orc.chunk_pool(x["k"]), sel)
    O_ref, lse_ref = orc.attend(x["q"], x["k"], x["v"], sel)
    O, lse = run.O.clone(), run.lse.clone()
    PU.assert_attention_close(PU.attention_errors(O.float().cpu().numpy().reshape(-1, d), lse.cpu().numpy().reshape(-1), O_ref, lse_ref))
    for again in range(30):                                # the work queue is rewound by the pass before
        run.attend_only()
        assert torch.equal(O, run.O) and torch.equal(lse, run.lse), again
    run.backward()
    rows = W.sample_rows(wl, 64)
    dQ_g, dK_g, dV_g = (t.float().cpu().numpy() for t in (run.dQ, run.dK, run.dV))
    off = wl.layout.chunk_off
    for head, chunk in ((0, 1), (heads - 1, wl.n_chunks // 2)):
        t0, t1 = int(off[chunk]), int(off[chunk + 1])
        dQ, dK, dV = orc.attend_bwd(x["q"], x["k"], x["v"], x["do"], sel, rows, head, (t0, t1))
        PU.assert_grad_close(dQ_g[rows[:, 0], rows[:, 1]], dQ)
        PU.assert_grad_close(dK_g[head, t0:t1], dK)
        PU.assert_grad_close(dV_g[head, t0:t1], dV)


@pytest.mark.parametrize("name,heads", [("mini2", 3), ("mini5", 2), ("midi2", 2), ("mini2", 5)])
def test_launches_that_overlap_leave_complete_results(name, heads):
    """A kernel that starts before the one in front of it is done: what follows in the stream, with no synchronisation in
    between, still finds every result, and finds the same bits each time."""
    wl = W.workload(name)
    wl.n_heads = heads
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do"))
    if heads > 3:                                          # room for the partials of two heads: groups of 2, 2, 1
        run.plan.moc_plan_set_workspace_budget(run.plan.workspace_bytes(False) - 3 * 2 * wl.n_tokens * wl.top_k * wl.head_dim)
        run.ws = run.g.empty((run.plan.workspace_bytes(True),), torch.uint8)
    run.forward().backward()
    p, x = run.plan, run.x
    outs = (run.O, run.lse, run.dQ, run.dK, run.dV)
    want, got = [t.clone() for t in outs], []
    for _ in range(12):
        for t in outs:
            t.fill_(float("nan"))
        p.moc_attend(x["q"], x["k"], x["v"], run.sel, run.O, run.lse, run.ws)
        p.moc_attend_bwd(x["q"], x["k"], x["v"], run.O, run.lse, x["do"], run.sel, run.dQ, run.dK, run.dV, run.ws)
        got.append([t.clone() for t in outs])
    run.check_status()
    for again, ts in enumerate(got):
        for a, b in zip(want, ts):
            assert torch.equal(a, b), again


@pytest.mark.parametrize("k", [9, 16, 17, 24, 31, 40])
def test_a_nan_score_is_never_picked(k):
    """Keys with a NaN make their chunk's descriptor NaN for every query of the head: the picks are what the clean stream gives
    without that chunk (from a list one longer); a query with a NaN picks nothing."""
    lay = W.make_layout(3, 8, 24, 33)                          # 72 score columns, the chunk among the first 32
    wl = W.Workload("nan", 2, 64, lay, k, 1, 1)
    longer = PU.GpuRun(W.Workload("nan", 2, 64, lay, k + 1, 1, 1)).forward().sel
    run, chunk, row = PU.GpuRun(wl), 5, lay.n_tokens - 3
    clean = run.forward().sel.clone()
    t0, t1 = int(lay.chunk_off[chunk]), int(lay.chunk_off[chunk + 1])
    run.x["k"][1, t0 + 1, 7] = float("nan")
    run.x["q"][0, row, 3] = float("nan")
    p = run.plan
    p.moc_chunk_pool(run.x["k"], run.desc, run.ws)
    p.moc_route(run.x["q"], run.desc, run.sel, run.ws)
    run.check_status()
    assert not bool((run.sel[1] == chunk).any()) and bool((clean[1] == chunk).any())
    want = torch.full_like(run.sel[1], -1)
    kept = longer[1] != chunk
    for i in range(lay.n_tokens):
        picks = longer[1, i][kept[i]][:k]
        want[i, :len(picks)] = picks
    assert torch.equal(run.sel[1], want)
    assert bool((run.sel[0, row] == -1).all())


@pytest.mark.parametrize("frames,causal", [(1, True), (7, True), (15, False), (16, True), (17, True), (31, False), (32, True)])
@pytest.mark.parametrize("k", [1, 4, 8])
def test_scores_that_are_not_numbers_among_few_chunks(frames, causal, k):
    """Up to 32 score columns and 8 picks, where the three terms of a score are added up by the selection: queries and keys with a NaN or an
    infinity, or whose scores overflow.  No score that is not a number is picked, and no chunk that is not a candidate."""
    lay = W.make_layout(1, 5, frames, 9)
    for spoil in ("nan query", "nan key", "inf key", "overflow"):
        run = PU.GpuRun(W.Workload("few", 2, 64, lay, k, 0, 0, causal=causal))
        p, q, key = run.plan, run.x["q"], run.x["k"]
        run.forward()
        clean = run.sel.clone()
        if spoil == "nan query":
            q[:, ::3, 7] = float("nan")
        elif spoil == "nan key":
            key[:, 5 + 9 * (frames // 2), 3] = float("nan")
        elif spoil == "inf key":
            key[:, 5 + 9 * (frames // 2), 3] = float("inf")
        else:
            q.mul_(2.0 ** 70)
            key.mul_(2.0 ** 70)
        p.moc_chunk_pool(key, run.desc, run.ws)
        p.moc_route(q, run.desc, run.sel, run.ws)
        run.check_status()
        sel = run.sel.cpu().numpy()
        own = lay.token_chunk()[None, :, None]
        assert np.all((sel >= -1) & (sel < lay.n_chunks) & (sel != 0) & (sel != own) & ((sel < own) if causal else True)), spoil
        ordered = np.sort(np.where(sel < 0, 10 ** 6 + np.arange(k), sel), axis=2)
        assert np.all(ordered[..., 1:] > ordered[..., :-1]), spoil                        # none twice
        if spoil == "nan query":
            assert np.all(sel[:, ::3] == -1) and torch.equal(run.sel[:, 1::3], clean[:, 1::3])
        elif spoil in ("nan key", "inf key"):
            assert not np.any(sel == 1 + frames // 2)         # (an infinite key's terms add up to no number)
