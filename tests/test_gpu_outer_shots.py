"""Scores of whole shots: as many as a block takes at a time, one more, one fewer, and several times as many."""
import numpy as np
import pytest
import torch

from paper_2508_21058_b200 import MocError, MocPlan
from paper_2508_21058_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", (64, 128))
@pytest.mark.parametrize("shots,caption,frames", [(2, 5, 1), (7, 3, 8), (8, 0, 9), (9, 40, 7), (17, 9, 17), (30, 1, 2)])
def test_every_shot(shots, caption, frames, d):
    wl = W.Workload("shots", 2, d, W.make_layout(shots, caption, frames, 37), 1, 1, 1)
    plan = MocPlan.from_workload(wl)
    ws, M, q0 = plan.new_workspace(), shots - 1, plan.L - 37 * frames
    x = torch.randn(2, plan.L, d, device="cuda", generator=torch.Generator("cuda").manual_seed(shots)).bfloat16()
    desc = torch.empty(2, plan.C, d, device="cuda")
    shot_desc, scores, sel = torch.empty(2, shots, d, device="cuda"), torch.empty(2, shots, device="cuda"), torch.empty(2, M, dtype=torch.int32, device="cuda")
    plan.moc_chunk_pool(x, desc, ws)
    plan.moc_outer_route(x, desc, q0, plan.L, M, shot_desc, scores, sel, ws)
    want = x.double().view(2, shots, -1, d).mean(2)
    # sums of at most n terms of size about 1 in fp32, each step half an ulp: n 2^-24, and as much again for the chunks' own means
    n = plan.L // shots
    assert float((shot_desc - want).abs().max()) < 2 * n * 2 ** -24
    xg = x[:, q0:].double().mean(1)
    assert float((scores - (want * xg[:, None]).sum(2)).abs().max()) < 4 * (n + d) * 2 ** -24
    left = scores[:, :M].clone()                             # the block is the last shot
    assert torch.equal(sel.long(), torch.argsort(left, dim=1, descending=True, stable=True))


@pytest.mark.parametrize("d,most", [(64, 12224), (128, 12160)])
def test_as_many_shots_as_the_header_states(d, most):
    """Shots of one token.  One more than the limit is refused before anything is written."""
    for S in (most, most + 1):
        lay = W.Layout(np.arange(S + 1, dtype=np.int32), np.arange(S, dtype=np.int32), np.zeros(S, np.uint8))
        plan = MocPlan.from_workload(W.Workload("shots", 1, d, lay, 1, 0, 0))
        x = torch.randn(1, S, d, device="cuda", generator=torch.Generator("cuda").manual_seed(d)).bfloat16()
        ws, desc, M = plan.new_workspace(), x.float(), 5
        shot_desc, scores, sel = torch.full((1, S, d), 7.0, device="cuda"), torch.full((1, S), 7.0, device="cuda"), torch.full((1, M), 7, dtype=torch.int32, device="cuda")
        if S > most:
            ws.fill_(9)
            with pytest.raises(MocError) as e:
                plan.moc_outer_route(x, desc, S - 300, S, M, shot_desc, scores, sel, ws)
            torch.cuda.synchronize()
            assert e.value.code == -2 and all(bool((t == 7).all()) for t in (shot_desc, scores, sel)) and bool((ws == 9).all())
            continue
        plan.moc_outer_route(x, desc, S - 300, S, M, shot_desc, scores, sel, ws)
        want = (x[0].double() * x[0, S - 300:].double().mean(0)).sum(1)
        # means of 300 terms and sums of d products of size about 1 in fp32, half an ulp each
        assert torch.equal(shot_desc, desc) and float((scores[0] - want).abs().max()) < (300 + d) * 2 ** -22
        assert torch.equal(sel[0].long(), torch.argsort(scores[0, :S - 300], descending=True, stable=True)[:M])
