"""Routing on scores that are too small for normal numbers, of both signs: they count as equal to zero and to each other, and every query
still gets as many picks as it has candidates for."""
import numpy as np
import pytest
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_chunks,k", [(20, 4), (20, 8), (60, 3), (60, 6), (100, 16), (120, 24), (300, 8), (300, 24), (300, 60), (700, 118)])
@pytest.mark.parametrize("sign", [-1, 0, 1])
def test_as_many_picks_as_there_are_candidates(n_chunks, k, sign):
    lay = W.Layout((3 * np.arange(n_chunks + 1)).astype(np.int32), np.zeros(n_chunks, np.int32), np.zeros(n_chunks, np.uint8))
    plan = MocPlan.from_workload(W.Workload("small", 2, 64, lay, k, 0, 0))
    gen = torch.Generator("cuda").manual_seed(k)
    q, key = (2.0 ** -68 * torch.randn(2, plan.L, 64, device="cuda", generator=gen) for _ in range(2))
    if sign:
        q, key = q.abs(), sign * key.abs()                       # scores of one sign, or of both
    ws, desc, sel = plan.new_workspace(), torch.empty(2, plan.C, 64, device="cuda"), torch.empty(2, plan.L, k, dtype=torch.int32, device="cuda")
    plan.moc_chunk_pool(key.bfloat16(), desc, ws)
    plan.moc_route(q.bfloat16(), desc, sel, ws)
    torch.cuda.synchronize()
    assert plan.moc_get_status(ws)[0] == 0
    own = torch.arange(plan.L, device="cuda") // 3               # the candidates: the chunks before the query's own
    assert torch.equal((sel >= 0).sum(2), own.clamp(max=k).expand(2, -1))
    assert bool((sel < own[None, :, None]).all())
    ordered = sel.masked_fill(sel < 0, 1 << 20).sort(2).values
    assert bool(((ordered[..., 1:] > ordered[..., :-1]) | (ordered[..., 1:] == 1 << 20)).all())       # no chunk twice
