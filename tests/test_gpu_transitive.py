"""TransitiveReduction (Alg. 1, Sec. 2) on the GPU (cg_transitive_reduction)
against the oracle, entry for entry (row offsets, columns, codes, suffixes),
and against the interval property at the 100 Mb size: the reduction of every
exact overlap among reads of one genome is the consecutive-overlap graph.
The reduced graph then goes through the contig path on the device."""
import numpy as np
import pytest

import gen
import oracle
from paper_2207_04350_gb300 import cg
from tests import _pins
from tests._gpu import assert_parity, run_gpu

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


def same_csr(a, b):
    for k in ("row_ptr", "col", "code", "suf"):
        x, y = np.asarray(getattr(a, k)), np.asarray(getattr(b, k))
        if x.shape != y.shape or not np.array_equal(x.astype(np.int64), y.astype(np.int64)):
            return False
    return True


def test_hand_cases(ctx):
    rows = [((1, 1, 1), (10, 15, 25, 30, 20, 50), 0), ((1, 1, 0), (10, 15, 25, 30, 20, 50), 0),
            ((1, 0, 1), (10, 15, 25, 30, 20, 50), 0), ((1, 1, 3), (10, 15, 25, 30, 20, 50), 0),
            ((1, 1, 1), (10, 15, 26, 30, 20, 51), 0), ((1, 1, 1), (10, 15, 26, 30, 20, 51), 1),
            ((1, 1, 1), (10, 15, 26, 30, 20, 50), 0), ((3, 2, 3), (10, 15, 25, 30, 20, 50), 0)]
    for codes, sufs, fuzz in rows:
        G = _pins._tr_triangle(*codes, *sufs)
        assert same_csr(cg.cg_transitive_reduction(ctx, G, fuzz), oracle.transitive_reduction(G, fuzz))


@pytest.mark.parametrize("fuzz", [0, 40])
def test_generated_with_repeats(ctx, fuzz):
    cfgs = [dict(gen.WORKLOADS["tiny-1Mb"](), full_overlaps=1),
            dict(gen._cfg(91, 600_000, [(0.08, 2000, 6000, 3, 10, 0.0)], 15, 1, 7000, 3000, 2500), full_overlaps=1),
            dict(gen._cfg(92, 800_000, [(0.1, 3000, 8000, 2, 12, 0.05)], 20, 0, 5000, 15000, 2500),
                 full_overlaps=1, rep_div_accept=0.1)]
    for d in cfgs:
        R = gen.generate(d, threads=8, off_align=1)
        S = cg.cg_transitive_reduction(ctx, R, fuzz)
        assert S.m < R.m
        assert same_csr(S, oracle.transitive_reduction(R, fuzz))


def test_noisy_suffixes(ctx):
    R = gen.generate(dict(gen.WORKLOADS["tiny-1Mb"](), full_overlaps=1), threads=8)
    rng = np.random.default_rng(3)
    N = type("N", (), {})()
    for k in ("row_ptr", "col", "code", "len", "off", "packed"):
        setattr(N, k, getattr(R, k))
    lv = np.asarray(R.len)[np.asarray(R.col)]
    N.suf = np.clip(np.asarray(R.suf) + rng.integers(-3, 4, size=R.m), 1, lv - 1).astype(np.int32)
    for fuzz in (0, 2, 6):
        assert same_csr(cg.cg_transitive_reduction(ctx, N, fuzz), oracle.transitive_reduction(N, fuzz))


def test_interval_property_100mb(ctx):
    d = dict(gen.WORKLOADS["genome-100Mb"](), k_rep=0)
    full = gen.generate(dict(d, full_overlaps=1), threads=16)
    red = gen.generate(d, threads=16)
    assert full.m > 3 * red.m
    S = cg.cg_transitive_reduction(ctx, full)
    assert same_csr(S, red)


def test_on_device_to_contigs(ctx):
    import torch
    R = gen.generate(dict(gen.WORKLOADS["tiny-1Mb"](), full_overlaps=1), threads=8)
    dev = type("D", (), {})()
    for k in ("row_ptr", "col", "code", "suf", "len", "off", "packed"):
        setattr(dev, k, torch.from_numpy(np.ascontiguousarray(getattr(R, k))).cuda())
    S = cg.cg_transitive_reduction(ctx, dev, device=True)
    S.len, S.off, S.packed = dev.len, dev.off, dev.packed
    host = type("H", (), {})()
    for k in ("row_ptr", "col", "code", "suf"):
        setattr(host, k, getattr(S, k).cpu().numpy())
    host.len, host.off, host.packed = R.len, R.off, R.packed
    assert same_csr(host, oracle.transitive_reduction(R))
    orc = oracle.run(host, min_chain_reads=2)
    g = cg.cg_load_graph(ctx, S, flags=cg.BORROW_DEVICE, min_chain_reads=2)
    try:
        off, bases = cg.contigs_host(g)
    finally:
        g.close()
    assert np.array_equal(off, orc.contig_off) and np.array_equal(bases, orc.bases)


def random_overlaps(seed, n, pairs, hub=0, hubs=(0,), clique=0):
    """Overlaps of random pairs among n reads, codes at random, suffixes of 1 to 4
    bases (so that many two-step walks add up); with `hub`, each of the reads `hubs`
    overlaps that many others, with `clique` the first so many reads all overlap."""
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, size=(2, pairs))
    for h in hubs if hub else ():
        others = np.delete(np.arange(n), h)[:hub]
        u, v = np.concatenate([u, np.full(hub, h)]), np.concatenate([v, others])
    if clique:
        a, b = np.triu_indices(clique, 1)
        u, v = np.concatenate([u, a]), np.concatenate([v, b])
    keep = u != v
    key = np.unique(np.minimum(u, v)[keep] * n + np.maximum(u, v)[keep])
    u, v = key // n, key % n
    code = rng.integers(0, 4, size=len(u))
    suf = rng.integers(1, 5, size=(2, len(u)))
    rows, cols = np.concatenate([u, v]), np.concatenate([v, u])
    codes = np.concatenate([code, ((code & 1) << 1) | (code >> 1)])
    sufs = np.concatenate(suf)
    o = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, rows + 1, 1)
    G = type("R", (), {})()
    G.row_ptr, G.col, G.code = np.cumsum(rp), cols[o].astype(np.int32), codes[o].astype(np.uint8)
    G.suf, G.len = sufs[o].astype(np.int32), np.full(n, 400, np.int32)
    G.off, G.packed, G.n, G.m = np.arange(n, dtype=np.int64) * 400, np.zeros(100 * n, np.uint8), n, len(cols)
    return G


@pytest.mark.parametrize("n,pairs,hub", [
    (1, 0, 0), (31, 15, 0), (33, 300, 0),       # no entries; a word of reads; dense rows
    (121, 2000, 0), (240, 3600, 0),             # batches of rows: 30 entries a row, so fewer rows than a batch holds
    (5000, 900, 0), (9000, 60, 0),              # mostly empty rows, batches that are not full
    (300, 12000, 0),                            # 80 entries a row
    (2600, 4000, 1530), (2600, 4000, 1545),     # a row about as long as what the walks stage
    (2600, 4000, 2040), (2600, 4000, 2500),     # a row about as long as, and longer than, what is staged
])
def test_row_shapes(ctx, n, pairs, hub):
    G = random_overlaps(n + hub, n, pairs, hub)
    for fuzz in (0, 1):
        assert same_csr(cg.cg_transitive_reduction(ctx, G, fuzz), oracle.transitive_reduction(G, fuzz))


@pytest.mark.parametrize("n,pairs,hub,hubs,clique", [
    (2600, 1500, 768, (0,), 0), (2600, 1500, 769, (0,), 0),     # as long as a piece, and one entry more
    (2600, 1500, 1535, (7,), 0), (2600, 1500, 1536, (7,), 0), (2600, 1500, 1537, (7,), 0),   # two pieces
    (3000, 1500, 2999, (0, 1, 2, 1500, 2999), 0),               # long rows side by side, the last read's too
    (9000, 30, 8999, (4000,), 0),                               # a long row among rows of one entry
    (1500, 0, 0, (), 150), (2000, 3000, 0, (), 400),            # rows of 149 and 400 entries side by side
])
def test_rows_in_pieces(ctx, n, pairs, hub, hubs, clique):
    G = random_overlaps(n + hub, n, pairs, hub, hubs, clique)
    for fuzz in (0, 1):
        assert same_csr(cg.cg_transitive_reduction(ctx, G, fuzz), oracle.transitive_reduction(G, fuzz))


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("n,pairs,hub,hubs,clique", [
    (200_000, 900, 0, (), 0), (20_000, 20_000, 0, (), 0), (300, 12000, 0, (), 0),
    (3000, 1500, 2999, (0, 1, 1500, 2999), 0), (2000, 3000, 0, (), 400)])
def test_scratch_within_a_tight_budget(n, pairs, hub, hubs, clique, device):
    """With 12 bytes of scratch per read and 6 per entry (and the copies of host arrays),
    too few for the rows' records and runs, the call gives the same."""
    import torch
    G = random_overlaps(n + hub, n, pairs, hub, hubs, clique)
    want = oracle.transitive_reduction(G, 1)
    k = len(want.col)
    arrays = [4 * G.m, G.m, G.m, 4 * n, 8 * (n + 1), 8, 8 * (n // 2048 + 3)]
    if not device:
        arrays += [8 * (n + 1), 4 * G.m, G.m, 4 * G.m, 4 * n, 4 * k, k, 4 * k]
    D = G
    if device:
        D = type("D", (), {})()
        for f in ("row_ptr", "col", "code", "suf", "len", "off", "packed"):
            setattr(D, f, torch.from_numpy(np.ascontiguousarray(getattr(G, f))).cuda())
    ctx = cg.cg_create(0, hbm_budget_bytes=sum((b + 255) // 256 * 256 for b in arrays))
    try:
        S = cg.cg_transitive_reduction(ctx, D, 1, device=device)
        for f in ("row_ptr", "col", "code", "suf"):
            got = getattr(S, f)
            assert np.array_equal(got.cpu().numpy() if device else got, getattr(want, f))
    finally:
        ctx.close()


def test_missing_or_foreign_mirrors(ctx):
    """An entry whose pair lacks the entry back, seen from the smaller and from the
    larger read, and one that leads to a read without entries."""
    G = random_overlaps(5, 200, 900)
    rows = np.repeat(np.arange(200), np.diff(G.row_ptr))
    for x in (np.flatnonzero(rows < G.col)[7], np.flatnonzero(rows > G.col)[11]):
        H = type("R", (), dict(vars(G)))()
        keep = np.arange(G.m) != x
        H.row_ptr = G.row_ptr - (np.arange(201) > rows[x])
        H.col, H.code, H.suf, H.m = G.col[keep], G.code[keep], G.suf[keep], G.m - 1
        with pytest.raises(cg.CgError) as e:
            cg.cg_transitive_reduction(ctx, H)
        assert e.value.status == cg.CG_EGRAPH
    H = type("R", (), dict(vars(G)))()
    H.row_ptr, H.col = np.append(G.row_ptr, G.m), G.col.copy()
    H.col[G.row_ptr[200] - 1], H.len = 200, np.full(201, 400, np.int32)
    H.off = np.arange(201, dtype=np.int64) * 400
    with pytest.raises(cg.CgError) as e:
        cg.cg_transitive_reduction(ctx, H)
    assert e.value.status == cg.CG_EGRAPH


def test_entries_without_reads(ctx):
    """Entries of a graph that has no reads: refused as an invalid graph, whatever the
    offsets say, and the context goes on."""
    G = random_overlaps(5, 200, 900)
    for rp in ([0], [3], [G.m]):
        H = type("R", (), dict(vars(G)))()
        H.row_ptr, H.len, H.off, H.n = np.array(rp, np.int64), G.len[:0], G.off[:0], 0
        with pytest.raises(cg.CgError) as e:
            cg.cg_transitive_reduction(ctx, H)
        assert e.value.status == cg.CG_EGRAPH
        assert same_csr(cg.cg_transitive_reduction(ctx, G), oracle.transitive_reduction(G))


@pytest.mark.parametrize("hub", [0, 1600])
@pytest.mark.parametrize("flip", [1, 2, 3])
def test_pairs_whose_ends_disagree(ctx, hub, flip):
    """One entry's code changed, seen from either read, in a row of any kind."""
    G = random_overlaps(9, 1800, 4000, hub)
    rows = np.repeat(np.arange(1800), np.diff(G.row_ptr))
    for x in (0, np.flatnonzero(rows < G.col)[-1], G.m - 1):
        H = type("R", (), dict(vars(G)))()
        H.code = G.code.copy()
        H.code[x] ^= flip
        with pytest.raises(cg.CgError) as e:
            cg.cg_transitive_reduction(ctx, H)
        assert e.value.status == cg.CG_EGRAPH


def test_invalid_and_capacity(ctx):
    G = _pins._tr_triangle(1, 1, 1, 10, 15, 25, 30, 20, 50)
    bad = []
    for k, i, v in (("col", 0, 2), ("col", 0, 9), ("code", 0, 4), ("suf", 0, 0)):
        H = type("H", (), {})()
        for f in ("row_ptr", "col", "code", "suf", "len", "off", "packed"):
            setattr(H, f, np.array(getattr(G, f), copy=True))
        getattr(H, f if False else k)[i] = v
        bad.append(H)
    for H in bad:
        with pytest.raises(cg.CgError) as e:
            cg.cg_transitive_reduction(ctx, H)
        assert e.value.status == cg.CG_EGRAPH
    import ctypes
    from paper_2207_04350_gb300.cg import _desc, lib
    d = _desc(G, 2)
    rp = np.empty(4, np.int64)
    small = np.empty(1, np.int32), np.empty(1, np.uint8), np.empty(1, np.int32)
    cnt = ctypes.c_int64(-1)
    st = lib().cg_transitive_reduction(ctx.ptr, ctypes.byref(d), 0, rp.ctypes.data, small[0].ctypes.data,
                                       small[1].ctypes.data, small[2].ctypes.data, 1, cg.MEM_HOST, ctypes.byref(cnt))
    assert st == cg.CG_EINVAL and cnt.value == 4
    S = cg.cg_transitive_reduction(ctx, G)         # still usable
    assert S.m == 4
