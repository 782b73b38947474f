"""dQ around the last key tile of a chunk: how many of its columns are formed, and how many steps of 16 keys the product takes."""
import pytest
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W

import parity_utils as PU
from test_gpu_backward_full import REL, _off

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", (64, 128))
@pytest.mark.parametrize("tail", (1, 16, 17, 48, 49, 64, 65, 80, 113, 127))
def test_dq_of_a_tile_of_few_keys(tail, d):
    """REL: bf16 rounding of P, dS and the results; a step of 16 of at most 13 x 16 keys left out would be off by sqrt(1 / 13) = 0.28,
    and the key of a one-key tile, of 130 in a chunk, by 0.09."""
    wl = W.Workload("tails", 2, d, W.make_layout(2, tail, 5, 128 + tail), 3, 1, 1)
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
    x = run.x
    ref = MocPlan.from_workload(wl, scalar_attend=True)
    ws = ref.new_workspace(with_bwd=True)
    ref.moc_lists_from_sel(run.sel, ws)
    want = [torch.empty_like(run.O) for _ in range(3)]
    ref.moc_attend_bwd(x["q"], x["k"], x["v"], run.O, run.lse, x["do"], run.sel, *want, ws)
    run.backward()
    for what, a, b in zip(("dQ", "dK", "dV"), (run.dQ, run.dK, run.dV), want):
        assert _off(a, b) < REL, what
