"""Graphs small enough for one block to run their mask, chain and offsets stages,
against the oracle, and the same graphs padded with reads without overlaps until
they take the kernels of larger graphs: every form of input, stage by stage and
as one deferred step, at the edges of words, of the block's threads and of the
rule that chooses."""
from types import SimpleNamespace

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


def step(ctx, G, mcr):
    """The whole step with nothing asked of its first stages, twice (captured, replayed)."""
    import torch
    dev = SimpleNamespace(**{k: torch.from_numpy(np.ascontiguousarray(getattr(G, k))).cuda()
                             if getattr(G, k, None) is not None else None
                             for k in ("row_ptr", "col", "code", "suf", "len", "off", "packed", "pre", "post")})
    g = cg.cg_load_graph(ctx, dev, flags=cg.BORROW_DEVICE, min_chain_reads=mcr)
    try:
        n, total = cg.cg_emit_contigs(g)
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        bases = torch.zeros(max(total, 16), dtype=torch.uint8, device="cuda")
        for _ in range(3):
            off.zero_()
            bases.zero_()
            torch.cuda.synchronize()
            cg.cg_mask_branches(g, want_count=False)
            cg.cg_chains(g, want_counts=False)
            cg.cg_emit_contigs(g, off, bases, want_counts=False)
            cg.cg_sync(ctx)
        return off.cpu().numpy(), bases[:total].cpu().numpy()
    finally:
        g.close()


def both(ctx, G, mcr):
    orc = oracle.run(G, min_chain_reads=mcr)
    assert_parity(run_gpu(ctx, G, min_chain_reads=mcr), orc)
    off, bases = step(ctx, G, mcr)
    assert np.array_equal(off, orc.contig_off) and np.array_equal(bases, orc.bases)


@pytest.mark.parametrize("lone", [0, 20_000])            # one block; the kernels of larger graphs
@pytest.mark.parametrize("sizes,closed", [
    ([2], [False]), ([31, 1, 2], [False] * 3), ([3, 4, 5], [True] * 3),
    ([1024], [False]), ([1023, 2], [False, True]), ([513] * 4, [True, False] * 2),
    ([4100, 7, 2], [False, True, False]), ([3] * 1500, [i % 7 == 0 for i in range(1500)]),
])
def test_chains(ctx, sizes, closed, lone):
    G = structured(sum(sizes) + lone, sizes, closed=closed, lone=lone)
    both(ctx, G, 2)
    both(ctx, G, 3)


@pytest.mark.parametrize("sizes,closed", [
    ([1400], [False]), ([1400], [True]), ([340] * 4, [True, False] * 2),      # as many entries as one block takes
    ([3] * 600, [i % 7 == 0 for i in range(600)]), ([2] * 1400, [False] * 1400), ([1] * 900 + [7] * 150, [False] * 1050),
])
def test_chains_of_one_block(ctx, sizes, closed):
    G = structured(sum(sizes), sizes, closed=closed)
    assert G.m <= 3400 - G.n // 9
    for mcr in (1, 2, 3):
        both(ctx, G, mcr)


@pytest.mark.parametrize("mcr", [1, 2])
@pytest.mark.parametrize("n", [1, 32, 33, 1025, 4096, 4097, 16384, 16385])
def test_read_counts(ctx, n, mcr):
    q = min(n, 700)
    both(ctx, structured(n, [q] if q > 1 else [], lone=n - q if q > 1 else n), mcr)


@pytest.mark.parametrize("n,m", [(3060, 3060), (3062, 3062), (8000, 2510), (8000, 2514), (16384, 1578), (16384, 1582)])
def test_entry_counts(ctx, n, m):
    """On either side of the line that falls with the reads."""
    both(ctx, structured(m, [2] * (m // 2), lone=n - m), 2)


@pytest.mark.parametrize("lone", [0, 20_000])
@pytest.mark.parametrize("rp", [np.int32, np.int64])
@pytest.mark.parametrize("mcr", [1, 2])
def test_forms(ctx, lone, rp, mcr):
    """Row offsets of either width, branch reads and both overlap forms."""
    G = gen.generate(dict(gen.WORKLOADS["tiny-1Mb"](), seed=77), threads=4, off_align=1)
    pad = lambda a, fill: np.concatenate([a, np.full(lone, fill, a.dtype)])  # noqa: E731
    H = SimpleNamespace(row_ptr=pad(np.asarray(G.row_ptr), G.m).astype(rp), col=G.col, code=G.code, suf=G.suf,
                        len=pad(G.len, 5), off=pad(G.off, 3), packed=G.packed, pre=None, post=None)
    both(ctx, H, mcr)
    pre, post = gen.xdrop_form(G, max_trim=300, seed=5, consistent=False)
    both(ctx, SimpleNamespace(**{**vars(H), "suf": None, "pre": pre, "post": post}), mcr)


def test_many_entries(ctx):
    """Few reads with more overlaps than one block takes: rows of up to 40."""
    rng = np.random.default_rng(3)
    pairs = {(min(a, b), max(a, b)) for a, b in rng.integers(0, 600, size=(6000, 2)) if a != b}
    ent = []
    for a, b in pairs:
        c = int(rng.integers(0, 4))
        ent += [(a, b, c, int(rng.integers(1, 9))), (b, a, ((c & 1) << 1) | (c >> 1), int(rng.integers(1, 9)))]
    ln, off, packed = gen.pack_reads(["ACGTTGCAAC"] * 640)
    rp, col, code, suf = gen.csr_from_entries(640, ent)
    assert len(col) > 8192
    both(ctx, SimpleNamespace(row_ptr=rp, col=col, code=code, suf=suf, len=ln, off=off, packed=packed), 1)
