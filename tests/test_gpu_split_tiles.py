"""dK and dV of a caption whose key tiles are shared by several blocks, against the CUDA-core kernels on the same selection: every
element, and the same bits whichever block is last."""
import pytest
import torch

from paper_2508_21058_b200 import MocPlan
from paper_2508_21058_b200 import workloads as W
from paper_2508_21058_b200.binding import debug_shared_key_tiles

import parity_utils as PU
from test_shared_key_tiles import LONG_CHUNK

pytestmark = pytest.mark.gpu

# heads, head_dim, (shots, caption, frames, frame length), k, blocks that share a caption's tile on 148 SMs
SHAPES = {
    "4 blocks, a tile of two rows": (2, 128, (1, 130, 24, 100), 2, 4),
    "8 blocks, two captions of 5": (1, 128, (2, 5, 40, 129), 1, 8),
    "8 blocks, three captions of two tiles": (1, 128, (3, 130, 30, 129), 3, 8),
    "6 blocks, one key": (1, 64, (1, 1, 40, 64), 2, 6),
    "7 blocks, d 64": (3, 64, (1, 40, 64, 97), 3, 7),
    "no room for the sums of two captions": (1, 128, (2, 5, 20, 129), 1, 1),
    "no room for their sums": (1, 128, (1, 140, 30, 100), 0, 1),           # without picks there are no partials to take the place of
}
# P and dS are rounded to bf16 (half an ulp: 2^-9) on one side, the results on both: a few 1e-3 of the 2-norm of a block of rows
# (seen: 4e-3).  Of at most 94 query tiles one left out, or taken twice, is off by sqrt(1 / 94) = 0.10.
REL = 2e-2


def check_every_gradient(wl, passes, spoil=None):
    run = PU.GpuRun(wl, tensors=("q", "k", "v", "do")).forward()
    x, outs = run.x, []
    ref = MocPlan.from_workload(wl, scalar_attend=True)
    ws = ref.new_workspace(with_bwd=True)
    ref.moc_lists_from_sel(run.sel, ws)
    want = [torch.empty_like(run.O) for _ in range(3)]
    ref.moc_attend_bwd(x["q"], x["k"], x["v"], run.O, run.lse, x["do"], run.sel, *want, ws)
    for _ in range(passes):
        if spoil:
            spoil.backward()
        run.backward()
        outs.append([t.clone() for t in (run.dQ, run.dK, run.dV)])
    off = wl.layout.chunk_off
    for got in outs:
        for a, b, first in zip(got, want, outs[0]):
            assert torch.equal(a, first)
            for c in range(wl.n_chunks):
                rows = slice(int(off[c]), int(off[c + 1]))
                diff, norm = ((t[:, rows].float()).flatten(1).norm(dim=1) for t in (a.float() - b.float(), b))
                assert float((diff / norm.clamp(min=1e-3)).max()) < REL, (c, float((diff / norm).max()))


@pytest.mark.parametrize("shape", SHAPES)
def test_every_gradient_of_a_shared_tile(shape):
    heads, d, lay, k, blocks = SHAPES[shape]
    wl = W.Workload("split", heads, d, W.make_layout(*lay), k, 1, 1)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert n_sm != 148 or set(debug_shared_key_tiles(wl, n_sm)[1]) == {blocks}
    check_every_gradient(wl, 20)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("stream", LONG_CHUNK)
def test_a_long_chunk_with_fewer_query_tiles_than_the_caption_has_blocks(stream, d):
    """After the backward of another stream, which leaves sums in every SM's tensor memory."""
    other = PU.GpuRun(W.Workload("spoil", 8, d, W.make_layout(1, 64, 12, 512), 2, 1, 1), tensors=("q", "k", "v", "do")).forward()
    check_every_gradient(LONG_CHUNK[stream](d), 3, other)
