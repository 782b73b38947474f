"""Every element of dQ, dK and dV (and of O) against the library's CUDA-core kernels over the same selection, on shapes of few
tiles, where one wrong tile of a block stands out, with dO read from DRAM: it is evicted from L2 before each call."""
import pytest
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU

pytestmark = pytest.mark.gpu

ALL = W.WHOLE_SHOT
# heads, head_dim, layout (shots, caption, frames, frame[, chunk]), k, back, fwd, causal, selection edited
SHAPES = {
    "ragged frames, three shots": (3, 128, (3, 40, 5, 200), 3, 1, 1, True, False),
    "64-token frames, d 64": (8, 64, (2, 16, 12, 64), 7, 1, 1, True, False),
    "64-token frames, d 128": (4, 128, (2, 30, 20, 64), 12, 1, 1, True, True),
    "whole tiles": (2, 128, (2, 128, 8, 128), 4, 1, 1, True, False),
    "windows of 256, not causal, d 64": (4, 64, (1, 77, 1, 3000, 256), 5, 0, 0, False, False),
    "not causal, d 128": (2, 128, (1, 50, 14, 190), 6, 0, 0, False, True),
    "512-token frames": (1, 128, (2, 64, 6, 512), 2, 1, 1, True, False),
    "one row past a tile": (5, 128, (2, 1, 11, 129), 9, 1, 1, True, False),
    "40 picks": (2, 128, (3, 8, 24, 40), 40, 0, 0, True, True),
    "one pick": (6, 64, (4, 100, 3, 333), 1, 2, 0, True, False),
    "whole shots": (2, 128, (5, 20, 4, 150), 3, ALL, ALL, True, True),
    "items of 256 and 128 rows": (7, 64, (2, 10, 9, 384), 6, 1, 1, True, False),
    "no picks": (3, 128, (2, 130, 3, 129), 0, 1, 1, True, False),
    "one chunk": (1, 128, (1, 0, 1, 100), 2, 0, 0, True, False),
}
# P, dS, the routed partials and the results are rounded to bf16 (half an ulp: 2^-9) on one side and not on the other: at most
# four such steps on a sum whose terms may cancel, a few 1e-3 of the 2-norm (seen: 4e-3 over 128 rows).  A tile of another
# step in one of n (here at most 80) is off by sqrt(2 / n) > 0.15.
REL = 2e-2


def _off(a, b):
    """The largest relative 2-norm of the difference over blocks of 128 rows of a head."""
    pad = (0, 0, 0, -a.shape[1] % 128)
    d, r = (torch.nn.functional.pad(t.float(), pad).unflatten(1, (-1, 128)).flatten(2).norm(dim=2) for t in (a.float() - b.float(), b))
    assert bool(torch.isfinite(a.float()).all())
    return float((d / r.clamp(min=1e-3)).max())


@pytest.mark.parametrize("shape", SHAPES)
def test_every_gradient_element(shape):
    heads, d, lay, k, back, fwd, causal, edited = SHAPES[shape]
    flush = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")          # twice the L2
    for seed in range(3):
        wl = W.Workload("every", heads, d, W.make_layout(*lay), k, back, fwd, causal, seed=seed)
        run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
        if edited:
            run.plan.moc_context_drop(run.sel, 0.5, 1.0, 17 + seed, run.ws)
            run.attend_only()
        x, outs = run.x, []
        ref = MocPlan.from_workload(wl, scalar_attend=True)
        ws = ref.new_workspace(with_bwd=True)
        ref.moc_lists_from_sel(run.sel, ws)
        O, lse = torch.empty_like(run.O), torch.empty_like(run.lse)
        ref.moc_attend(x["q"], x["k"], x["v"], run.sel, O, lse, ws)
        assert _off(run.O, O) < REL
        want = [torch.empty_like(run.O) for _ in range(3)]
        ref.moc_attend_bwd(x["q"], x["k"], x["v"], run.O, run.lse, x["do"], run.sel, *want, ws)
        for again in range(3):
            flush.fill_(again)
            run.backward()
            outs.append([t.clone() for t in (run.dQ, run.dK, run.dV)])
        for got in outs:
            for what, a, b in zip(("dQ", "dK", "dV"), got, want):
                assert _off(a, b) < REL, (what, seed)
                assert torch.equal(a, outs[0][("dQ", "dK", "dV").index(what)]), (what, seed)
