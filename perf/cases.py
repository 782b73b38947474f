"""The workloads that the library's speed is followed on: complete passes of the path (pool -> route -> attend, with its
backward, the training-time edits of the selection, and the shot-level pre-selection) through the public entry points.

A case is a dict of plain values:
    task      "forward"; "train" (forward and backward); "drop" (train, with context drop-off / drop-in between routing and
              attention); "outer" (shots pre-selected for the last shot's queries, then a forward pass on the reduced stream)
    heads, dim, k, causal, back, fwd      the plan's parameters; back / fwd: the intra-shot window, -1 = the whole shot
    shots, caption, frames, frame, chunk  the token layout: per shot a caption chunk and frames * frame video tokens, cut into
              frames (chunk = 0) or into windows of `chunk` tokens with a short last one
    repeats   in how many shots a frame's content comes back (0: every chunk has content of its own)
    top_m     shots to select ("outer" only, else 0)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W

P_MAX, LAMBDA = 0.5, 1.0          # the context drop-off / drop-in setting of the tests


def _case(task, heads, dim, shots, caption, frames, frame, chunk, k, back, fwd, causal=True, repeats=0, top_m=0, **name):
    return dict(name, task=task, heads=heads, dim=dim, shots=shots, caption=caption, frames=frames, frame=frame, chunk=chunk, k=k,
                back=back, fwd=fwd, causal=causal, repeats=repeats, top_m=top_m)


def listed():
    return [
        # a few hundred tokens: the first steps of a progressive schedule, debugging runs; launches and latency are all of it
        _case("forward", 4, 64, 1, 64, 8, 64, 0, 2, 0, 0, name="small-clip-fwd"),
        # a small training step with ragged frames, three shots
        _case("train", 3, 128, 3, 40, 5, 200, 0, 3, 1, 1, name="small-scenes-train"),
        # the single-shot variant: not causal, every chunk of 256 tokens sees itself and the prompt; head_dim 64
        _case("train", 12, 64, 1, 77, 1, 6240, 256, 5, 0, 0, causal=False, name="single-shot-noncausal-train"),
        # a middle-sized training step with the selection regularised; an odd frame length
        _case("drop", 8, 128, 4, 128, 9, 1170, 0, 4, 1, 1, name="scenes-drop-train"),
        # one clip of 33k tokens, all heads: inference and training
        _case("forward", 24, 128, 1, 256, 21, 1560, 0, 4, 0, 0, name="clip-fwd"),
        _case("train", 24, 128, 1, 256, 21, 1560, 0, 4, 0, 0, name="clip-train"),
        # eight shots, 264k tokens, all heads: the largest inference pass
        _case("forward", 24, 128, 8, 256, 21, 1560, 0, 6, 1, 1, name="scenes-fwd"),
        # the same stream in finer chunks, where many chunks are picked per query (a device's share of the heads)
        _case("forward", 6, 128, 8, 256, 21, 1560, 512, 32, 1, 1, repeats=4, name="scenes-chunk512-fwd"),
        _case("forward", 6, 128, 8, 256, 21, 1560, 256, 30, 1, 1, repeats=4, name="scenes-chunk256-fwd"),
        _case("forward", 2, 128, 8, 256, 21, 1560, 256, 118, 1, 1, repeats=4, name="scenes-chunk256-dense-fwd"),
        # a training step on a minute of video, 528k tokens (a device's share of the heads)
        _case("train", 4, 128, 16, 256, 21, 1560, 0, 8, 1, 1, name="minute-train"),
        # generation of the last shot of eight: three earlier shots pre-selected, then the pass on the reduced stream
        _case("outer", 4, 128, 8, 256, 21, 1560, 0, 6, 1, 1, top_m=3, name="outer-then-fwd"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: clips and multi-shot streams of 500 to 530k tokens, frames or windows of 64 to 2048 tokens, 1 to 118 picks."""
    while True:
        task = rng.choice(["forward", "forward", "forward", "forward", "train", "train", "train", "drop", "outer"])
        clip = task != "outer" and rng.random() < 0.35
        shots = 1 if clip else _log_int(rng, 3 if task == "outer" else 2, 16)
        c = _case(task, _log_int(rng, 1, 24), 64 if rng.random() < 0.25 else 128, shots, _log_int(rng, 16, 256), _log_int(rng, 4, 40),
                  _log_int(rng, 64, 1560), 0 if rng.random() < 0.5 else _log_int(rng, 64, 2048), _log_int(rng, 1, 118),
                  *rng.choice([(0, 0), (1, 1), (1, 1), (2, 0), (W.WHOLE_SHOT, W.WHOLE_SHOT)]),
                  causal=not (clip and rng.random() < 0.3), repeats=0 if clip or rng.random() < 0.5 else 4,
                  top_m=rng.randint(1, shots - 1) if task == "outer" else 0)
        if clip and c["back"] == W.WHOLE_SHOT:
            c["back"] = c["fwd"] = 0                   # a clip that attends to all of itself routes nothing
        if c["chunk"] > c["frames"] * c["frame"] // 2:
            continue
        chunks = _layout(c).n_chunks - shots
        c["k"] = min(c["k"], max(1, chunks // 3))
        while c["heads"] > 1 and not _affordable(c):
            c["heads"] //= 2
        if _affordable(c):
            return c


def _affordable(c):
    L, C = _layout(c).n_tokens, _layout(c).n_chunks
    if c["heads"] * L * C * 2 > 8e9 or L * c["k"] * c["dim"] * 2 > 2e9 or c["heads"] * L * c["dim"] * 2 > 2e9:
        return False
    # short chunks and heads of 64 run at a lower rate: a drawn case shall not take longer than the largest listed one
    return work(c)["flops"] * max(1.0, 512 / (c["chunk"] or c["frame"])) * (128 / c["dim"]) < 1.5e13


def _layout(c):
    return W.make_layout(c["shots"], c["caption"], c["frames"], c["frame"], c["chunk"] or None)


def _pairs(c, lay):
    """Selected (query, key) pairs of one head and scored (query, chunk) pairs: anchors by the rule, picks at the mean video chunk."""
    size, text, shot = np.diff(lay.chunk_off).astype(np.int64), lay.chunk_mod == 1, lay.chunk_shot
    idx = np.arange(lay.n_chunks)
    back, fwd = (lay.n_chunks if v == W.WHOLE_SHOT else v for v in (c["back"], c["fwd"]))
    mean_video = float(size[~text].mean())
    pairs = scored = 0.0
    for q in range(lay.n_chunks):
        anchor = text | ((shot == shot[q]) & (idx >= q - back) & (idx <= q + fwd))
        cand = ~anchor & ((idx < q) if c["causal"] else True)
        n = int(cand.sum())
        pairs += float(size[q]) * (float(size[anchor].sum()) + min(c["k"], n) * mean_video)
        scored += float(size[q]) * n
    return pairs, scored


def work(c):
    lay, H, d, k = _layout(c), c["heads"], c["dim"], c["k"]
    L, C = lay.n_tokens, lay.n_chunks
    row = 2.0 * H * L * d                                    # one bf16 tensor
    if c["task"] == "outer":
        # the features are read once for the shots' descriptors; attention then works on the kept shots alone
        kept = dict(c, task="forward", shots=c["top_m"] + 1)
        texts = c["shots"] - kept["shots"]                   # captions of the shots left out stay, as keys and as queries
        inner = work(kept)
        more = 2.0 * H * texts * c["caption"] * d
        return {"bytes": row + 2.0 * H * c["frames"] * c["frame"] * d + inner["bytes"] + 4 * more,
                "flops": inner["flops"] + 4.0 * d * H * texts * c["caption"] * (_layout(kept).n_tokens + texts * c["caption"])}
    pairs, scored = _pairs(c, lay)
    out = {"bytes": 4 * row + 4.0 * H * (L + C * d + L * k), "flops": H * (4.0 * d * pairs + 2.0 * d * scored)}
    if c["task"] != "forward":
        out["bytes"] += 4 * row                              # dO in, dQ, dK, dV out
        out["flops"] += H * 10.0 * d * pairs
    return out


def tolerance(c):
    # Against kernels that keep P and dS in fp32 and sum in another order (two heads of each case): O is off by 3.1e-3, the
    # gradients by at most 3.5e-3 in the 2-norm and 0.14 of their RMS at the worst value (dV of keys that few queries weigh);
    # against scores summed in fp64, up to 1.3e-5 of the picks differ (near ties).  Four times that.
    return {"rel": 1.4e-2, "max": 0.55, "differ": 5e-5}


def _inputs(c, seed, names):
    """bf16 [H][L][d] on the GPU: keys scattered around their chunk's centre, queries around the centre of a chunk that is
    drawn among those up to their own, values and output gradients without structure."""
    lay = _layout(c)
    wl = W.Workload("case", c["heads"], c["dim"], lay, c["k"], c["back"], c["fwd"], c["causal"], seed=seed % 65521,
                    shared_identities=c["repeats"])
    gen = torch.Generator("cuda").manual_seed(seed)
    ids = torch.from_numpy(W.centre_ids(wl)).cuda()
    tok = torch.from_numpy(lay.token_chunk().astype(np.int64)).cuda()
    H, L, d = c["heads"], lay.n_tokens, c["dim"]
    x = {n: torch.empty((H, L, d), dtype=torch.bfloat16, device="cuda") for n in names}
    noise = torch.empty((L, d), dtype=torch.float32, device="cuda")
    for h in range(H):
        centre = 0.5 * torch.randn((2 * lay.n_chunks + 1, d), generator=gen, device="cuda")[ids]
        aim = (torch.rand(L, generator=gen, device="cuda") * (tok + 1)).long().clamp(max=lay.n_chunks - 1)
        for n in names:
            noise.normal_(generator=gen)
            if n == "k":
                noise += centre[tok]
            elif n == "q":
                noise += centre[aim]
            x[n][h] = noise
    return wl, x


def prepare(c, seed):
    train = c["task"] in ("train", "drop")
    wl, x = _inputs(c, seed, ("q", "k", "v", "do") if train else ("q", "k", "v"))
    plan = MocPlan.from_workload(wl)
    return {"case": c, "x": x, "plan": plan, "ws": plan.new_workspace(with_bwd=train), "seed": seed}


def run(s):
    c, x, plan, ws = s["case"], s["x"], s["plan"], s["ws"]
    if c["task"] == "outer":
        return _run_outer(s)
    if c["task"] == "forward":
        return plan.forward(x["q"], x["k"], x["v"], ws)[:4]
    dev = x["q"].device
    if c["task"] == "train":
        desc, sel, O, lse, _ = plan.forward(x["q"], x["k"], x["v"], ws)
    else:
        desc = torch.empty((plan.H, plan.C, plan.d), dtype=torch.float32, device=dev)
        sel = torch.empty((plan.H, plan.L, plan.k), dtype=torch.int32, device=dev)
        O, lse = torch.empty_like(x["q"]), torch.empty((plan.H, plan.L), dtype=torch.float32, device=dev)
        plan.moc_chunk_pool(x["k"], desc, ws)
        plan.moc_route(x["q"], desc, sel, ws)
        plan.moc_context_drop(sel, P_MAX, LAMBDA, s["seed"], ws)
        plan.moc_attend(x["q"], x["k"], x["v"], sel, O, lse, ws)
    dQ, dK, dV = (torch.empty_like(x["q"]) for _ in range(3))
    plan.moc_attend_bwd(x["q"], x["k"], x["v"], O, lse, x["do"], sel, dQ, dK, dV, ws)
    return desc, sel, O, lse, dQ, dK, dV


def _run_outer(s):
    """The last shot's video tokens are the query block; the first stream's selection serves every stream."""
    c, x, plan, ws = s["case"], s["x"], s["plan"], s["ws"]
    dev, S = x["q"].device, plan.moc_outer_num_shots()
    q0, q1 = plan.L - c["frames"] * c["frame"], plan.L
    desc = torch.empty((plan.H, plan.C, plan.d), dtype=torch.float32, device=dev)
    shot_desc = torch.empty((plan.H, S, plan.d), dtype=torch.float32, device=dev)
    scores = torch.empty((plan.H, S), dtype=torch.float32, device=dev)
    sel_shot = torch.empty((plan.H, c["top_m"]), dtype=torch.int32, device=dev)
    plan.moc_chunk_pool(x["k"], desc, ws)
    plan.moc_outer_route(x["q"], desc, q0, q1, c["top_m"], shot_desc, scores, sel_shot, ws)
    off, shot, mod, tok = plan.moc_outer_reduced_layout(sel_shot[0].cpu().numpy(), q0, q1)
    tok_map = torch.from_numpy(tok).to(dev)
    red = [torch.empty((plan.H, len(tok), plan.d), dtype=torch.bfloat16, device=dev) for _ in range(3)]
    for src, dst in zip((x["q"], x["k"], x["v"]), red):
        plan.moc_gather_tokens(src, tok_map, dst)
    inner = MocPlan(plan.H, len(tok), plan.d, off, shot, mod, c["k"], c["back"], c["fwd"], c["causal"])
    out = inner.forward(*red)[:4]
    inner.close()
    return (shot_desc, scores, sel_shot, *red, *out)
