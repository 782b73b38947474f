"""The forward's routed partials, from where routed items leave them to where anchor items merge them, at the edges of their
layout and variants, against the CUDA-core attention kernels on the same selection."""
import pytest
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU

pytestmark = pytest.mark.gpu

# heads, head_dim, (shots, caption, frames, frame length), k, drop: chunks that start off and on the 128-query blocks of the layout,
# rows of a warp in two blocks, a warp and a query tile with a few rows or none
SHAPES = {
    "register merge, 1 pick": (2, 128, (2, 7, 6, 130), 1, False),
    "register merge, batches of 3 + 1": (2, 128, (2, 16, 9, 257), 4, False),
    "register merge, whole batches": (2, 128, (2, 31, 9, 161), 6, False),
    "register merge, empty slots": (2, 128, (2, 7, 12, 140), 7, True),
    "block copies, 1 pick": (1, 128, (2, 7, 6, 577), 1, False),
    "block copies, 2 picks": (1, 128, (2, 8, 6, 545), 2, False),          # as many as stages per block
    "block copies, 5 picks, empty slots": (1, 128, (2, 9, 10, 609), 5, True),
    "d 64, 1 pick": (2, 64, (2, 7, 6, 130), 1, False),
    "d 64, 2 picks, one loading warp": (2, 64, (2, 33, 7, 290), 2, False),
    "d 64, 3 picks": (2, 64, (2, 1, 9, 65), 3, False),                    # as many as stages
    "d 64, 4 picks, empty slots": (2, 64, (3, 5, 9, 129), 4, True),
    "d 64, 9 picks, one loading warp": (2, 64, (2, 3, 14, 300), 9, True),
    # more slots than chunks to pick: rows that use none, fewer than are asked for ahead, or some of them
    "register merge, 3 of 12 slots": (2, 128, (1, 16, 5, 130), 12, False),
    "register merge, 5 of 20 slots, some empty": (2, 128, (1, 16, 7, 140), 20, True),
    "block copies, 3 of 12 slots": (2, 128, (1, 16, 5, 577), 12, False),
    "block copies, 5 of 20 slots, some empty": (1, 128, (1, 16, 7, 530), 20, True),
    "d 64, 3 of 12 slots": (2, 64, (1, 16, 5, 130), 12, False),
    "d 64, 5 of 20 slots, some empty, one loading warp": (2, 64, (1, 16, 7, 300), 20, True),
}
# P and the partials are rounded to bf16 on one side and not on the other (half an ulp: 2^-9), as is O on both: three such steps, 6e-3,
# on the 2-norm of a block of rows; a slot missed, taken twice or weighed wrongly is off by more than a tenth (at most 9 picks).
REL = 2e-2


@pytest.mark.parametrize("shape", SHAPES)
def test_every_element_of_the_merge(shape):
    heads, d, lay, k, drop = SHAPES[shape]
    wl = W.Workload("merge", heads, d, W.make_layout(*lay), k, 1, 1)
    run = PU.GpuRun(wl).forward()
    if drop:
        run.plan.moc_context_drop(run.sel, 0.9, 0.5, 3, run.ws)
        assert bool((run.sel < 0).any())
    x = run.x
    ref = MocPlan.from_workload(wl, scalar_attend=True)
    ws = ref.new_workspace()
    ref.moc_lists_from_sel(run.sel, ws)
    O, lse = torch.empty_like(run.O), torch.empty_like(run.lse)
    ref.moc_attend(x["q"], x["k"], x["v"], run.sel, O, lse, ws)
    # what an empty slot's place holds must not matter
    for fill in (0xff, 0x00):
        run.ws.fill_(fill)
        run.plan.moc_lists_from_sel(run.sel, run.ws)
        run.attend_only()
        run.check_status()
        pad = (0, 0, 0, -run.O.shape[1] % 128)
        diff, norm = (torch.nn.functional.pad(t, pad).unflatten(1, (-1, 128)).flatten(2).norm(dim=2) for t in (run.O.float() - O.float(), O.float()))
        assert bool(torch.isfinite(run.O.float()).all())
        assert float((diff / norm.clamp(min=1e-3)).max()) < REL
        assert float((run.lse - lse).abs().max()) < 2e-3


@pytest.mark.parametrize("d,frame", [(64, 130), (64, 400), (128, 130), (128, 600)])
def test_tensors_on_16_byte_boundaries(d, frame):
    """Every tensor of the boundary is 16-byte aligned and no more: the same bits as with 256-byte aligned ones."""
    wl = W.Workload("align", 2, d, W.make_layout(2, 7, 6, frame), 3, 1, 1)
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()

    def off(t):
        flat = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
        assert flat.data_ptr() % 32 == 0
        return flat[8:].view(t.shape)

    x = {n: off(t).copy_(t) for n, t in run.x.items()}
    O, dQ, dK, dV = (off(run.O) for _ in range(4))
    lse, p = torch.empty_like(run.lse), run.plan
    p.moc_chunk_pool(x["k"], run.desc, run.ws)
    p.moc_route(x["q"], run.desc, run.sel, run.ws)
    run.attend_only()
    run.backward()                                             # on the same lists: their order is the order of sums
    p.moc_attend(x["q"], x["k"], x["v"], run.sel, O, lse, run.ws)
    p.moc_attend_bwd(x["q"], x["k"], x["v"], O, lse, x["do"], run.sel, dQ, dK, dV, run.ws)
    assert p.moc_get_status(run.ws)[0] == 0
    for a, b in ((O, run.O), (dQ, run.dQ), (dK, run.dK), (dV, run.dV)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("d,frame,k", [(128, 130, 3), (128, 600, 5), (64, 130, 3), (64, 400, 5)])
def test_weights_of_large_scores_sum_to_one(d, frame, k):
    """Scores with a common part of some 4e5: values of one come out as one.  The partials and O are sums of P rounded to bf16 over the
    sum of P (half an ulp each: 2^-9), so O is one or the bf16 below."""
    wl = W.Workload("large", 2, d, W.make_layout(1, 16, 16, frame), k, 0, 0)
    run = PU.GpuRun(wl)
    for n in ("q", "k"):
        run.x[n][..., 0] = 2000.0
    run.x["v"].fill_(1.0)
    run.forward()
    assert float(run.lse.min()) > 3e5
    assert float((run.O.float() - 1).abs().max()) <= 2 ** -8
