"""Which key tiles of dK/dV are shared by several blocks, and by how many (the rule of csrc/moc_plan.cu, through its host-only hook):
a block reads accumulators that it alone has written, so each must have a query tile."""
import numpy as np
import pytest

from paper_2508_21058_b200 import workloads as W
from paper_2508_21058_b200.binding import debug_shared_key_tiles

N_SM = 148


def ragged(heads, d, sizes, k, back=0, fwd=0, captions=(0,), shots=None):
    """A stream of chunks of these sizes; `captions` are its text chunks."""
    n = len(sizes)
    lay = W.Layout(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), np.asarray(shots if shots is not None else [0] * n, np.int32),
                   np.isin(np.arange(n), captions).astype(np.uint8))
    return W.Workload("ragged", heads, d, lay, k, back, fwd)


# streams in which a chunk is long beside its neighbours and has fewer query tiles than the caption has blocks
LONG_CHUNK = {
    "two query tiles": lambda d: ragged(1, d, [128] + [16] * 46 + [250], 12),
    "six query tiles": lambda d: ragged(1, d, [122] + [64] * 144 + [747], 7),
    "one query tile, last shot": lambda d: ragged(1, d, [64] + [8] * 300 + [16] * 3, 2, 1, 1, shots=[0] + list(range(300)) + [300] * 3),
}


@pytest.mark.parametrize("stream", LONG_CHUNK)
def test_a_long_chunk_has_no_more_blocks_than_query_tiles(stream):
    query_tiles, blocks, _ = debug_shared_key_tiles(LONG_CHUNK[stream](128), N_SM)
    assert query_tiles.min() < blocks.max()                    # the case: the caption's number would be too many
    assert np.all(blocks >= 1) and np.all(blocks <= query_tiles)


def test_every_block_has_a_query_tile_whatever_the_stream():
    rng, uneven = np.random.RandomState(0), 0
    for x in range(2000):
        n, size, window = rng.randint(10, 160), rng.choice([8, 16, 33, 64, 100]), (0, 0)
        sizes, captions, shots = np.full(n, size), (0,), None
        sizes[-1] *= rng.randint(2, 20)                      # equal chunks and a longer last one
        if x % 2:                                            # anything
            sizes = rng.randint(1, 2 * size, n)
            sizes[rng.randint(n, size=rng.randint(1, 4))] *= rng.randint(1, 20)
            captions = (0, n // 2) if rng.rand() < 0.5 else (0,)
            shots, window = np.sort(rng.randint(rng.choice([1, 3, n]), size=n)), rng.choice([0, 1, 3, W.WHOLE_SHOT], 2)
        sizes[list(captions)] = rng.choice([1, 5, 64, 128, 256, 1000])
        wl = ragged(rng.choice([1, 2, 4]), rng.choice([64, 128]), sizes, rng.choice([1, 2, 4, 9, 20]), *window, captions, shots)
        query_tiles, blocks, _ = debug_shared_key_tiles(wl, N_SM)
        assert np.all((blocks >= 1) & (blocks <= 8) & (blocks <= query_tiles)), (sizes, shots, query_tiles, blocks)
        # tiles first..last of block p: floor(n p / blocks) to floor(n (p + 1) / blocks), with n at least the query tiles
        for n_qt, b in zip(query_tiles, blocks):
            cuts = np.arange(b + 1) * int(n_qt) // int(b)
            assert np.all(np.diff(cuts) >= 1)
        uneven += len(blocks) > 0 and query_tiles.min() < blocks.max()
    assert uneven > 20


@pytest.mark.parametrize("heads,caption,chunks,size,n_sm", [(1, 5000, 30, 608, 148), (2, 6656, 30, 1560, 2000), (2, 12800, 30, 1560, 2000)])
def test_the_counters_of_shared_tiles_fit_their_area(heads, caption, chunks, size, n_sm):
    """A caption of many key tiles before few chunks: more counters than the stream has chunks, which the work queue follows."""
    query_tiles, blocks, room = debug_shared_key_tiles(ragged(heads, 128, [caption] + [size] * chunks, 4), n_sm)
    assert blocks.max() > 1 and len(blocks) > chunks + 1
    assert 4 * heads * len(blocks) <= room
