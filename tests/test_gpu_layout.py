"""The layout's scans at the edges of their tiles, against the oracle: contig
heads in tiles of 8,192 reads (lone reads fill whole words of the heads bitmap,
chain heads sit between them), pieces in tiles of 1,024 walk positions, and
more pieces than one look (256 tiles) of the look-back covers."""
import numpy as np
import pytest

import gen
import oracle
from paper_2207_04350_gb300 import cg
from tests._gpu import assert_parity, run_gpu
from tests._graphs import structured

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2207_04350_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()
    c = cg.cg_create(0)
    yield c
    c.close()


@pytest.mark.parametrize("sizes,lone,mcr", [
    ([], 1, 1), ([], 31, 1), ([], 33, 1),                               # a word of heads
    ([], 8191, 1), ([], 8192, 1), ([], 8193, 1), ([2, 5], 16384, 1),    # a tile of the heads bitmap
    ([1023], 0, 2), ([1024], 0, 2), ([1025], 0, 2),                     # a tile of pieces
    ([2] * 512, 9000, 2), ([2] * 513, 9000, 2),                         # heads in every other word
    ([3, 1, 2, 40, 1], 270_000, 1),                                     # 264 tiles of pieces
])
def test_tile_edges(ctx, sizes, lone, mcr):
    G = structured(len(sizes) + lone, sizes, lone=lone)
    assert_parity(run_gpu(ctx, G, min_chain_reads=mcr, inputs="device", outputs="device"),
                  oracle.run(G, min_chain_reads=mcr))


def test_heads_in_one_word(ctx):
    """Chains whose smallest reads are neighbours: several chain heads per word,
    with lone reads between them, in both minimum chain lengths."""
    G = structured(21, [2] * 3000, lone=50)
    for mcr in (1, 2):
        assert_parity(run_gpu(ctx, G, min_chain_reads=mcr), oracle.run(G, min_chain_reads=mcr))
    assert np.count_nonzero(oracle.run(G).contig_off) == 3000


@pytest.mark.parametrize("mb", [50, 90, 330])
def test_spelling_spans(mb):
    """Spans of 2, 4 and 16 tiles (on 608 warps) with smaller ones at the end,
    whole and in shares that start at any tile."""
    import torch
    G = gen.generate(dict(gen.WORKLOADS["genome-3.1Gb"](), genome_len=mb * 1_000_000), threads=8)
    want = oracle.run(G)
    c = cg.cg_create(0)
    try:
        cg.cg_set_tuning(c, emit_blocks_per_sm=1, emit_block_threads=128)
        assert_parity(run_gpu(c, G, inputs="device", outputs="device"), want)
        g = cg.cg_load_graph(c, G)
        for share in range(3):
            first, n = cg.cg_emit_share(g, share, 3)
            out = torch.full(((n + 15) // 16 * 16 + 16,), 7, dtype=torch.uint8, device="cuda")
            cg.cg_emit_share(g, share, 3, None, out)
            out = out.cpu().numpy()
            assert np.array_equal(out[:n], want.bases[first:first + n]) and (out[n:] == 7).all()
        g.close()
    finally:
        c.close()


@pytest.mark.parametrize("sizes,closed", [
    ([200_000, 40], [False, False]), ([700_000], [False]),             # jumped by two blocks per SM, and by more of them
    ([60_000, 300, 3], [True, False, True]), ([400_000], [True]),      # closed chains: by two per SM, and by all blocks
    ([90_000, 90_000], [False, True])])
def test_lists_that_a_part_of_the_grid_jumps(ctx, sizes, closed):
    G = structured(len(sizes), sizes, closed=closed, lone=50)
    want = oracle.run(G)
    for outputs in ("host", "device"):                                 # chains alone, then per-read outputs with them
        assert_parity(run_gpu(ctx, G, inputs="device", outputs=outputs), want)
