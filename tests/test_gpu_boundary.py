"""Contract of the C ABI beyond plain parity: a workspace that does not hold the plan's lists is refused
on the device without a fault, an edited selection is honoured after moc_lists_from_sel, a bounded wait
that runs out is reported and leaves the GPU usable, the workspace budget, and the debug build."""
import ctypes
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2508_21058_b200 import MocError, MocPlan
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ERR_WORKSPACE, ERR_TIMEOUT, ERR_TOO_LARGE = -5, -8, -9


def _outputs(plan, with_grads=False):
    O = torch.full((plan.H, plan.L, plan.d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((plan.H, plan.L), 7.0, dtype=torch.float32, device="cuda")
    return O, lse


@pytest.mark.parametrize("fill", [0, 0xA5])
def test_unrouted_workspace_is_refused_on_the_device(fill):
    """moc_attend / moc_attend_bwd on a workspace that moc_route never wrote (zero-filled, or full of a
    byte pattern): every block returns at once, nothing is written, the status says MOC_ERR_WORKSPACE."""
    wl = W.workload("mini2")
    x = W.generate(wl, "cuda", ("q", "k", "v", "do"))
    plan = MocPlan.from_workload(wl)
    ws = torch.full((plan.workspace_bytes(True),), fill, dtype=torch.uint8, device="cuda")
    ws[:64] = 0                                   # status words: no error recorded, no cookie
    sel = torch.full((plan.H, plan.L, plan.k), -1, dtype=torch.int32, device="cuda")
    O, lse = _outputs(plan)
    plan.moc_attend(x["q"], x["k"], x["v"], sel, O, lse, ws)
    torch.cuda.synchronize()
    assert plan.moc_get_status(ws)[0] == ERR_WORKSPACE
    assert bool(torch.all(O == 7.0)) and bool(torch.all(lse == 7.0))
    ws[:64] = 0
    grads = [torch.full_like(O, 7.0) for _ in range(3)]
    plan.moc_attend_bwd(x["q"], x["k"], x["v"], O, lse, x["do"], sel, *grads, ws)
    torch.cuda.synchronize()
    assert plan.moc_get_status(ws)[0] == ERR_WORKSPACE
    assert all(bool(torch.all(g == 7.0)) for g in grads)
    # the same workspace, once routed, works
    desc = torch.empty((plan.H, plan.C, plan.d), dtype=torch.float32, device="cuda")
    plan.moc_chunk_pool(x["k"], desc, ws)
    plan.moc_route(x["q"], desc, sel, ws)
    plan.moc_attend(x["q"], x["k"], x["v"], sel, O, lse, ws)
    torch.cuda.synchronize()
    assert plan.moc_get_status(ws)[0] == 0
    assert not bool(torch.any(O == 7.0).all())


def test_workspace_routed_by_another_plan_is_refused():
    wl_a, wl_b = W.workload("mini2"), W.workload("mini2t")     # same stream, another window: other lists
    wl_b.n_heads = wl_a.n_heads
    x = W.generate(wl_a, "cuda", ("q", "k", "v"))
    plan_a, plan_b = MocPlan.from_workload(wl_a), MocPlan.from_workload(wl_b)
    assert plan_a.workspace_bytes() == plan_b.workspace_bytes()
    ws = plan_a.new_workspace()
    desc, sel, O, lse, _ = plan_a.forward(x["q"], x["k"], x["v"], ws)
    torch.cuda.synchronize()
    assert plan_a.moc_get_status(ws)[0] == 0
    O2, lse2 = _outputs(plan_b)
    plan_b.moc_attend(x["q"], x["k"], x["v"], sel, O2, lse2, ws)
    torch.cuda.synchronize()
    assert plan_b.moc_get_status(ws)[0] == ERR_WORKSPACE
    assert bool(torch.all(O2 == 7.0))


def _edited_selection(wl, sel, rng):
    """A selection the router would not have produced: picks removed, picks swapped for other legal
    chunks, holes in the middle of a row, plus entries that must be dropped (an anchor, a future chunk,
    a repeat, an index out of range)."""
    lay = wl.layout
    tc = lay.token_chunk()
    H, L, k = sel.shape
    out = sel.copy()
    illegal = np.zeros_like(out, dtype=bool)
    for h in range(H):
        for i in rng.choice(L, L // 3, replace=False):
            c = int(tc[i])
            s = int(rng.randint(k))
            what = rng.randint(6)
            if what == 0:
                out[h, i, s] = -1                                   # a hole
            elif what == 1 and c > 0:
                out[h, i, s] = int(rng.randint(c))                  # any earlier chunk (may be an anchor or a repeat)
            elif what == 2:
                out[h, i, s] = c                                    # own chunk: an anchor
            elif what == 3 and c + 1 < lay.n_chunks:
                out[h, i, s] = c + 1                                # a future chunk
            elif what == 4:
                out[h, i, s] = lay.n_chunks + 5                     # out of range
            elif what == 5 and k > 1:
                out[h, i, s] = out[h, i, (s + 1) % k]               # a repeat
    return out


def _clean_like_the_contract(wl, orc, sel):
    """What moc_lists_from_sel must leave in sel_idx, written from the header's rule."""
    lay = wl.layout
    tc = lay.token_chunk()
    out = sel.copy()
    anchors = {}
    for h in range(sel.shape[0]):
        for i in range(sel.shape[1]):
            c = int(tc[i])
            if c not in anchors:
                anchors[c] = PU.anchor_chunks(orc, lay, c)
            seen = set()
            for s in range(sel.shape[2]):
                j = int(sel[h, i, s])
                ok = 0 <= j < lay.n_chunks and j not in anchors[c] and (j < c or not wl.causal) and j not in seen
                if ok:
                    seen.add(j)
                else:
                    out[h, i, s] = -1
    return out


# (repeats are found by comparing with up to 4 picks, by a bitmap of the row's picks with 12 and 20)
@pytest.mark.parametrize("name", ["mini2", "mini9", "mini5", "mini6", "mini10"])
def test_edited_selection_is_honoured_after_lists_from_sel(name):
    wl = W.workload(name)
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
    x = run.host_inputs()
    orc = Oracle.from_workload(wl)
    edited = _edited_selection(wl, run.sel.cpu().numpy(), np.random.RandomState(5))
    want = _clean_like_the_contract(wl, orc, edited)
    assert np.any(want != run.sel.cpu().numpy())
    run.sel.copy_(torch.from_numpy(edited).cuda())
    run.plan.moc_lists_from_sel(run.sel, run.ws)
    run.attend_only()
    sel_now = run.sel.cpu().numpy()
    assert np.array_equal(sel_now, want)                                       # illegal entries blanked, the rest untouched
    assert run.plan.moc_selected_pairs(run.ws) == orc.pair_count(want)
    O_ref, lse_ref = orc.attend(x["q"], x["k"], x["v"], want)
    err = PU.attention_errors(run.O.float().cpu().numpy().reshape(-1, wl.head_dim), run.lse.cpu().numpy().reshape(-1), O_ref, lse_ref)
    PU.assert_attention_close(err)
    # and the backward over the same edited selection
    run.backward()
    rows = W.sample_rows(wl, 48)
    lay = wl.layout
    chunk = 1
    t0, t1 = int(lay.chunk_off[chunk]), int(lay.chunk_off[chunk + 1])
    dQ, dK, dV = orc.attend_bwd(x["q"], x["k"], x["v"], x["do"], want, rows, 0, (t0, t1))
    PU.assert_grad_close(run.dQ.float().cpu().numpy()[rows[:, 0], rows[:, 1]], dQ)
    PU.assert_grad_close(run.dK.float().cpu().numpy()[0, t0:t1], dK, what="dK")
    PU.assert_grad_close(run.dV.float().cpu().numpy()[0, t0:t1], dV, what="dV")


def test_lists_from_sel_of_the_routers_own_selection_changes_nothing():
    wl = W.workload("mini2")
    run = PU.GpuRun(wl).forward()
    sel0, O0, lse0 = run.sel.clone(), run.O.clone(), run.lse.clone()
    pairs0 = run.plan.moc_selected_pairs(run.ws)
    run.plan.moc_lists_from_sel(run.sel, run.ws)
    run.attend_only()
    assert torch.equal(run.sel, sel0)
    assert run.plan.moc_selected_pairs(run.ws) == pairs0
    assert float((run.O.float() - O0.float()).abs().max()) <= 1e-2           # the same rows, grouped into other tiles
    assert float((run.lse - lse0).abs().max()) <= 1e-3


def test_a_wait_that_runs_out_is_reported_and_the_gpu_stays_usable():
    """A block waits on a barrier nothing arrives on, through the library's bounded wait with a 2 ms limit:
    it must give up, record MOC_ERR_TIMEOUT with the probe's code, and return; the attention kernels then
    refuse to start on that workspace (status set) until routing clears it, after which all is as before."""
    wl = W.workload("mini2")
    run = PU.GpuRun(wl).forward()
    O0 = run.O.clone()
    run.plan.debug_set_wait_limit_us(2000)
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    run.plan.debug_wait_probe(run.ws, 777)
    t1.record()
    torch.cuda.synchronize()
    assert 1.5 <= t0.elapsed_time(t1) <= 200.0                       # gave up after the stated limit, not the default second
    assert run.plan.moc_get_status(run.ws) == (ERR_TIMEOUT, 777)
    run.O.fill_(7.0)
    run.plan.moc_attend(run.x["q"], run.x["k"], run.x["v"], run.sel, run.O, run.lse, run.ws)
    torch.cuda.synchronize()
    assert bool(torch.all(run.O == 7.0))                             # a workspace with an error recorded runs nothing
    run.plan.debug_set_wait_limit_us(0)
    run.forward()                                                    # routing clears the status
    assert float((run.O.float() - O0.float()).abs().max()) <= 1e-2


@pytest.mark.parametrize("form", [0, 1, 2])
def test_every_form_of_wait_gives_up_after_its_limit(form):
    """A wait that parks, one that polls, one on a counter, each for something that never comes, with a limit of 4 ms."""
    run = PU.GpuRun(W.workload("mini2")).forward()
    run.plan.debug_set_wait_limit_us(4000)
    for code in (700, 701):                                      # (the first call loads the kernel)
        run.ws[:64] = 0
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        run.plan.debug_wait_probe(run.ws, code, form)
        t1.record()
        torch.cuda.synchronize()
        assert run.plan.moc_get_status(run.ws) == (ERR_TIMEOUT, code)
    assert 3.5 <= t0.elapsed_time(t1) <= 20.0                    # once to twice the limit as measured, and room for another clock


def test_workspace_budget_groups_heads_and_results_do_not_change():
    wl = W.workload("mini2")
    wl.n_heads = 5
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward().backward()
    full = run.plan.workspace_bytes(False)
    ref = [t.clone() for t in (run.sel, run.O, run.lse, run.dQ, run.dK, run.dV)]
    small = PU.GpuRun(wl, tensors=("q", "k", "v", "do"))
    per_head = 2 * wl.n_tokens * wl.top_k * wl.head_dim
    small.plan.moc_plan_set_workspace_budget(full - 3 * per_head)   # room for two heads' partials: groups of 2, 2, 1
    assert small.plan.workspace_bytes(False) <= full - 3 * per_head
    small.ws = small.g.empty((small.plan.workspace_bytes(True),), torch.uint8)
    small.forward().backward()
    got = (small.sel, small.O, small.lse, small.dQ, small.dK, small.dV)
    assert torch.equal(got[0], ref[0])
    for a, b in zip(got[1:], ref[1:]):
        assert float((a.float() - b.float()).abs().max()) <= 1e-2
    with pytest.raises(MocError) as e:
        small.plan.moc_plan_set_workspace_budget(per_head // 2)
    assert e.value.code == ERR_TOO_LARGE


def test_a_workspace_routed_under_another_budget_is_refused():
    """The work queue in the workspace is laid out by groups of heads: with other groups it is not followed."""
    wl = W.workload("mini2")
    wl.n_heads = 5
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
    want = run.O.clone()
    full = run.plan.workspace_bytes(False)
    run.plan.moc_plan_set_workspace_budget(full - 3 * 2 * wl.n_tokens * wl.top_k * wl.head_dim)      # groups of 2, 2, 1
    x, grads = run.x, [torch.full_like(run.O, 7.0) for _ in range(3)]
    run.O.fill_(7.0)
    run.plan.moc_attend(x["q"], x["k"], x["v"], run.sel, run.O, run.lse, run.ws)
    run.plan.moc_attend_bwd(x["q"], x["k"], x["v"], run.O, run.lse, x["do"], run.sel, *grads, run.ws)
    torch.cuda.synchronize()
    assert run.plan.moc_get_status(run.ws)[0] == ERR_WORKSPACE
    assert all(bool(torch.all(t == 7.0)) for t in (run.O, *grads))
    run.forward()                                                    # routed again, it works
    assert float((run.O.float() - want.float()).abs().max()) <= 1e-2


def test_debug_build_checks_every_workspace_index_and_finds_nothing():
    """The same sources built with -DMOC_DEBUG check every index taken from the workspace; on a sound run
    they must stay silent (status 0) and give the same answers.  Runs in a child process: a process loads
    one variant of the library."""
    code = (
        "import numpy as np, torch, sys\n"
        "sys.path.insert(0, %r); sys.path.insert(0, %r)\n"
        "import parity_utils as PU\n"
        "from oracle import Oracle\n"
        "from paper_2508_21058_b200 import workloads as W, lib_path\n"
        "assert lib_path().endswith('libmoc_debug.so')\n"
        "for name in ('mini2', 'mini9', 'mini7'):\n"
        "    wl = W.workload(name)\n"
        "    run = PU.GpuRun(wl, tensors=('q', 'k', 'v', 'do')).forward().backward()\n"
        "    x = run.host_inputs(); orc = Oracle.from_workload(wl)\n"
        "    sel = run.sel.cpu().numpy()\n"
        "    PU.assert_routing(wl, orc, x['q'], orc.chunk_pool(x['k']), sel)\n"
        "    O_ref, lse_ref = orc.attend(x['q'], x['k'], x['v'], sel)\n"
        "    PU.assert_attention_close(PU.attention_errors(run.O.float().cpu().numpy().reshape(-1, wl.head_dim), run.lse.cpu().numpy().reshape(-1), O_ref, lse_ref))\n"
        "    run.plan.moc_lists_from_sel(run.sel, run.ws); run.attend_only()\n"
        "print('DEBUG_BUILD_OK')\n"
    ) % (ROOT, os.path.join(ROOT, "tests"))
    from paper_2508_21058_b200 import build as libbuild
    libbuild.build(debug=True)                  # a no-op when libmoc_debug.so is up to date with the sources
    env = dict(os.environ, MOC_LIBRARY="debug", MOC_PARITY_DIR=os.path.join(PU.OUT_ROOT, "parity_debug"))
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, timeout=600)
    assert res.returncode == 0 and "DEBUG_BUILD_OK" in res.stdout, res.stdout[-2000:] + res.stderr[-4000:]


def test_many_short_items_in_a_row_never_wait_for_good():
    """256-token chunks with 30 picks per query: tens of thousands of attention items a few microseconds long, so that a
    CTA's softmax, its bookkeeping and its loads drift apart as far as the hand-overs between them allow."""
    wl = W.workload("cfg3-m256-p8")
    wl.n_heads = 2
    run = PU.GpuRun(wl).forward()
    O, lse = run.O.clone(), run.lse.clone()
    for _ in range(20):
        run.ws.random_(0, 256)
        run.forward()                                                # checks the device status
        assert torch.equal(O, run.O) and torch.equal(lse, run.lse)


@pytest.mark.parametrize("name", ["mini2", "cfg1"])              # tables of 20 KB, and of 150 KB
def test_a_new_plans_tables_are_there_for_a_stream_of_any_kind(name):
    """A plan made while the copy engine is busy, and used at once on a non-blocking stream."""
    wl = W.workload(name)
    wl.n_heads = 2
    x = W.generate(wl, "cuda", ("q", "k", "v"))
    want = MocPlan.from_workload(wl).forward(x["q"], x["k"], x["v"])[:4]
    host, dev = torch.empty(1 << 28, dtype=torch.uint8, pin_memory=True), torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    copies, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    plans = []                                                   # closing one would wait for the whole device
    for _ in range(6):
        with torch.cuda.stream(copies):
            for _ in range(4):
                dev.copy_(host, non_blocking=True)
        plan = MocPlan.from_workload(wl)
        plans.append(plan)
        with torch.cuda.stream(side):
            *got, ws = plan.forward(x["q"], x["k"], x["v"])
            assert plan.moc_get_status(ws)[0] == 0               # waits for the side stream alone
            assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_plans_are_made_in_every_context_of_the_device():
    """A plan's tables go over on a stream that is kept; a stream belongs to one context.  (Only made and destroyed in the second one:
    the tensors of this process belong to the first.)"""
    cu, ctx, wl = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), W.workload("mini2")
    before = PU.GpuRun(wl).forward()
    assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, torch.cuda.current_device()) == 0
    try:
        for _ in range(2):
            MocPlan.from_workload(wl).close()
    finally:
        assert cu.cuCtxDestroy_v2(ctx) == 0
    after = PU.GpuRun(wl).forward()
    for n in ("desc", "sel"):
        assert torch.equal(getattr(before, n), getattr(after, n)), n
    assert float((before.O.float() - after.O.float()).abs().max()) <= 1e-2          # the same rows, grouped into other tiles


@pytest.mark.parametrize("k,calls", [(4, 20000), (40, 3000)])
def test_plans_of_different_sizes_route_from_several_threads(k, calls):
    """One kernel serves plans whose tables take different amounts of shared memory; a thread's call may come between another's
    preparation and its launch.  (With the size of the plan as the kernel's attribute one launch in 6000 failed.)"""
    runs, failed = [], []
    for n_chunks in (60, 60, 600, 600):
        lay = W.Layout(np.arange(n_chunks + 1, dtype=np.int32), np.zeros(n_chunks, np.int32), (np.arange(n_chunks) == 0).astype(np.uint8))
        wl = W.Workload("threads", 1, 64, lay, k, 0, 0)
        plan, x = MocPlan.from_workload(wl), W.generate(wl, "cuda", ("q", "k"))
        ws, desc = plan.new_workspace(), torch.empty((1, plan.C, 64), dtype=torch.float32, device="cuda")
        sel = torch.empty((1, plan.L, k), dtype=torch.int32, device="cuda")
        plan.moc_chunk_pool(x["k"], desc, ws)
        plan.moc_route(x["q"], desc, sel, ws)
        runs.append((plan, x["q"], desc, sel, ws, sel.clone()))
    torch.cuda.synchronize()

    def many(plan, q, desc, sel, ws, _):
        stream = torch.cuda.Stream()
        args = (plan._h, *(t.data_ptr() for t in (q, desc, sel, ws)), stream.cuda_stream)
        for n in range(calls):
            code = plan._lib.moc_route(*args)                    # (as bare as can be: the threads shall meet inside the call)
            if code:
                failed.append((n, code))
            if n % 256 == 0:
                stream.synchronize()

    threads = [threading.Thread(target=many, args=r) for r in runs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for plan, q, desc, sel, ws, want in runs:
        assert plan.moc_get_status(ws)[0] == 0 and torch.equal(sel, want)
