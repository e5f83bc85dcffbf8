"""The work that programs have this library do, as cases that can be timed and compared.

A program loads string graphs, masks the branch reads, finds the chains and
spells the contigs; it reduces overlap graphs, partitions contigs, splits the
spelling over ranks and serves requests. Every case goes through the binding's
public calls, as such a program makes them. The graphs are drawn on the GPU
from the seed: reads sampled from a genome with lognormal lengths, contained
reads kept without overlaps, an overlap between each pair of consecutive
uncontained reads that share 2 kb or more, and overlaps between random pairs
of reads, as repeats cause them, which make branch reads. Read lengths,
coverages and genome sizes are those of the repository's workloads. The bases
themselves are random: no step of the library compares them.

All outputs are whole numbers and bytes, so every tolerance is "exact" and
there is no 64-bit form to compare with.
"""
import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2207_04350_gb300 import cg

MIN_OVERLAP = 2000

# One context and one server for the process, as a program keeps them: its graphs share a stream and a memory pool.
_kept = {}


def _context():
    if "ctx" not in _kept:
        _kept["ctx"] = cg.cg_create(0)
    return _kept["ctx"]


def _server():
    if "server" not in _kept:
        _kept["server"] = cg.Server(workers=8, max_batch=64, hbm_budget_bytes=60 << 30)
    return _kept["server"]


# ---------------------------------------------------------------- the cases
def _step(name, genome, **more):
    return {"name": name, "kind": "step", "genome": genome, "coverage": 30, "mean": 12000, "sd": 6000, "out": "ascii",
            "form": "suffix", "min_chain": 2, "row_bytes": 4, "align": 32, **more}


def _other(name, kind, genome, **more):
    return {"name": name, "kind": kind, "genome": genome, "coverage": 30, "mean": 12000, "sd": 6000, **more}


def listed():
    return [
        # one bacterial-size graph, the smallest call: mask, chains and ASCII contigs into device buffers
        _step("step-1Mb", 1_000_000, coverage=10, mean=10000, sd=3000),
        # an ordinary eukaryote: the same calls on 333k reads
        _step("step-100Mb", 100_000_000, coverage=40),
        # a human-size genome, the largest: 6.2M reads, int64 row offsets
        _step("step-3.1Gb", 3_100_000_000, mean=15000, sd=8000, row_bytes=8),
        # contigs kept packed, a quarter of the bytes, at an odd size
        _step("step-2bit-1.2Gb", 1_234_567_891, mean=15000, sd=8000, out="2bit", row_bytes=8),
        # the aligner's (pre, post) overlaps, lone reads spelled too, reads at any 4-base offset
        _step("step-xdrop-lone-37Mb", 37_654_321, form="xdrop", min_chain=1, align=4),
        # where every read went: branch flags, chain ids, ranks and orientations per read, and no spelling
        _other("reads-500Mb", "reads", 500_000_000, min_chain=2),
        # many uneven graphs of one load spelled in one pass
        _other("batch-512", "batch", 12_000_000, mean=10000, sd=5000, graphs=512),
        # one graph from pinned host memory to contigs in host memory: loaded and checked, spelled, freed
        _other("request-42Mb", "request", 42_000_000),
        # requests of 1 to 20 Mb through the server, submitted together
        _other("serve-24", "serve", 20_000_000, graphs=24),
        # the overlap graph before reduction: 3.4M entries among 6.2M reads
        _other("reduce-3.1Gb", "reduce", 3_100_000_000, mean=15000, sd=8000),
        # contigs to 72 processes by their reads
        _other("partition-72", "partition", 3_100_000_000, mean=15000, sd=8000, parts=72, weight=0),
        # one rank of eight that each hold an eighth of the reads: sizes, packing, spelling what was received
        _other("exchange-8", "exchange", 1_000_000_000, mean=15000, sd=8000, ranks=8),
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm, mostly odd."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["reads", "batch", "request", "serve", "reduce", "partition", "exchange"])
    mean = rng.choice([10000, 12000, 15000])
    if kind == "step":
        c = _step("", _log(rng, 300_000, 3_000_000_000), mean=mean, out=rng.choice(["ascii", "ascii", "2bit"]),
                  form=rng.choice(["suffix", "suffix", "xdrop"]), min_chain=rng.choice([2, 2, 2, 3, 1]),
                  row_bytes=rng.choice([4, 8]), align=rng.choice([32, 32, 4, 1]))
        if c["min_chain"] == 1:        # every lone read is spelled: the output is then as large as the reads
            c["genome"] = _log(rng, 300_000, 90_000_000)
    elif kind == "reads":
        c = _other("", kind, _log(rng, 1_000_000, 2_000_000_000), mean=mean, min_chain=rng.choice([1, 2, 3]))
    elif kind == "batch":
        c = _other("", kind, _log(rng, 1_000_000, 12_000_000), mean=mean, graphs=_log(rng, 8, 512))
    elif kind == "request":
        c = _other("", kind, _log(rng, 1_000_000, 100_000_000), mean=mean)
    elif kind == "serve":
        c = _other("", kind, _log(rng, 1_500_000, 30_000_000), mean=mean, graphs=rng.randint(2, 31))
    elif kind == "reduce":
        c = _other("", kind, _log(rng, 1_000_000, 3_000_000_000), mean=mean)
    elif kind == "partition":
        c = _other("", kind, _log(rng, 10_000_000, 3_000_000_000), mean=mean, parts=_log(rng, 2, 1024),
                   weight=rng.choice([0, 0, 1]))
    else:
        c = _other("", kind, _log(rng, 10_000_000, 1_000_000_000), mean=mean, ranks=rng.randint(2, 16))
    c["sd"] = mean // 2
    del c["name"]
    return c


# ---------------------------------------------------------------- the inputs
def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _graph(case, seed, genome=None, full=False, bases=True):
    """One string graph on the GPU: row_ptr, col, code, suf, len, off and packed. With `full` every pair of
    uncontained reads sharing 2 kb has its overlap, not the consecutive ones alone."""
    dev, r = "cuda", _rng(seed)
    G = int(genome or case["genome"])
    n = _reads(case, G)
    s2 = math.log(1 + (case["sd"] / case["mean"]) ** 2)
    length = torch.exp(torch.randn(n, device=dev, generator=r, dtype=torch.float64) * math.sqrt(s2) +
                       (math.log(case["mean"]) - s2 / 2)).long().clamp_(MIN_OVERLAP, min(G - 1, (1 << 20) - 1))
    start = (torch.rand(n, device=dev, generator=r, dtype=torch.float64) * (G - length + 1).double()).long()
    key = start * (1 << 20) + ((1 << 20) - 1 - length)            # by start, the longer read first
    order = torch.sort(key).indices
    start, length = start[order], length[order]
    end = start + length
    before = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), torch.cummax(end, 0).values[:-1]])
    kept = torch.nonzero(end > before).view(-1)                   # uncontained: starts and ends both increase
    rid = torch.randperm(n, device=dev, generator=r)              # read ids in no order of place
    strand = torch.randint(0, 2, (n,), device=dev, generator=r)
    k = kept.numel()
    ka, ke, kl = start[kept], end[kept], length[kept]
    # true overlaps: a is left through its right end, b entered through its left one
    ia, ib = [], []
    for step in range(1, k):
        i = torch.nonzero(ke[:k - step] - ka[step:] >= MIN_OVERLAP).view(-1)
        if i.numel() == 0:
            break
        ia.append(i)
        ib.append(i + step)
        if not full:
            break
    a = torch.cat(ia) if ia else torch.zeros(0, dtype=torch.int64, device=dev)
    b = torch.cat(ib) if ib else a
    ov = ke[a] - ka[b]
    ea, eb = 1 - strand[kept[a]], strand[kept[b]]
    # overlaps that repeats cause: a random end of one read with a random end of another
    m = max(1, int(2.3e-6 * G)) if k > 8 else 0
    x, y = (torch.randint(0, max(1, k), (m,), device=dev, generator=r) for _ in range(2))
    ex, ey = (torch.randint(0, 2, (m,), device=dev, generator=r) for _ in range(2))
    short = torch.minimum(kl[x], kl[y]) - 1 if m else x
    ok = (x != y) & (short > MIN_OVERLAP) if m else x > 0
    u01 = torch.rand(m, device=dev, generator=r, dtype=torch.float64)
    rov = MIN_OVERLAP + (u01 * (short - MIN_OVERLAP + 1).double()).long().clamp_(min=0)
    x, y, ex, ey, rov = x[ok], y[ok], ex[ok], ey[ok], torch.minimum(rov, short)[ok]
    a, b, ea, eb, ov = (torch.cat(p) for p in ((a, x), (b, y), (ea, ex), (eb, ey), (ov, rov)))
    # one overlap per pair of reads, the true one first
    pair = torch.minimum(a, b) * max(1, k) + torch.maximum(a, b)
    pair, at = torch.sort(pair, stable=True)
    first = torch.ones_like(pair, dtype=torch.bool)
    first[1:] = pair[1:] != pair[:-1]
    at = at[first]
    a, b, ea, eb, ov = a[at], b[at], ea[at], eb[at], ov[at]
    u, v = rid[kept[a]], rid[kept[b]]
    src, dst = torch.cat([u, v]), torch.cat([v, u])
    code = torch.cat([ea | (eb << 1), eb | (ea << 1)])
    suf = torch.cat([kl[b] - ov, kl[a] - ov])
    at = torch.sort(src * n + dst).indices
    rows = torch.bincount(src, minlength=n)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(rows, 0, out=row_ptr[1:])
    by_id = torch.empty_like(length)
    by_id[rid] = length
    align = case.get("align", 32)
    room = (by_id + align - 1) // align * align
    off = torch.cumsum(room, 0) - room
    nbytes = (int(room.sum()) + 63) // 64 * 16
    packed = None
    if bases:
        packed = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        packed.view(torch.int32).random_(-2**31, 2**31 - 1, generator=r)
    g = SimpleNamespace(row_ptr=row_ptr if case.get("row_bytes", 4) == 8 else row_ptr.int(), col=dst[at].int(),
                        code=code[at].to(torch.uint8), suf=suf[at].int(), len=by_id.int(), off=off, packed=packed,
                        packed_bytes=nbytes, pre=None, post=None)
    if case.get("form") == "xdrop":
        _xdrop(g, src[at], r)
    return g


def _xdrop(g, u, r, most=200):
    """The (pre, post) form of g's exact overlaps, each reported up to `most` bases late on either read."""
    v, code, length = g.col.long(), g.code.long(), g.len.long()
    lu, lv = length[u], length[v]
    ov = lv - g.suf.long()
    slack = torch.full((length.numel(),), 1 << 40, dtype=torch.int64, device=length.device)
    slack.scatter_reduce_(0, u, lu - ov - 1, "amin")
    cap = torch.minimum(torch.clamp(ov - 1, max=most), slack[v]).clamp_(min=0)
    tu, tv = ((torch.rand(u.numel(), device=u.device, generator=r, dtype=torch.float64) * (cap + 1).double()).long()
              for _ in range(2))
    pre = lu - ov - 1 + tu
    g.pre = torch.where((code & 1) == 1, pre, lu - 1 - pre).int()
    g.post = torch.where((code >> 1) == 0, tv, lv - 1 - tv).int()
    g.suf = None


def _sizes(case):
    """Genome sizes of a pool's graphs: log-uniform up to the case's, over a factor of twenty."""
    r = np.random.default_rng(7)
    lo, hi = math.log(max(300_000, case["genome"] / 20)), math.log(case["genome"])
    return [int(math.exp(r.uniform(lo, hi))) for _ in range(case["graphs"])]


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _to_host(g):
    fields = {k: _pinned(getattr(g, k)) for k in ("row_ptr", "col", "code", "suf", "len", "off", "packed")}
    return SimpleNamespace(pre=None, post=None, **fields)


def _zeros(count, dtype=torch.uint8, **where):
    """An output buffer; what a pass does not write of it stays zero."""
    return torch.zeros(max(1, int(count)), dtype=dtype, **(where or {"device": "cuda"}))


def _reads(case, genome=None):
    return max(4, int(case["coverage"] * int(genome or case["genome"]) / case["mean"]))


def _room(case, genome=None):
    """What the outputs of a graph are sized for: contig offsets, contig bases."""
    genome = int(genome or case["genome"])
    if case.get("min_chain") == 1:                    # every read may be a contig of its own
        return _reads(case, genome) + 1, int(1.1 * case["coverage"] * genome) + 2_000_000
    return _reads(case, genome) // 2 + 2, int(1.25 * genome) + 2_000_000


def _fits(sizes, room):
    if sizes[0] + 1 > room[0] or sizes[1] > room[1]:
        raise RuntimeError(f"outputs of {sizes} do not fit {room}")


def prepare(case, seed):
    kind, ctx = case["kind"], _context()
    s = {"case": case}
    if kind in ("step", "reads", "partition"):
        s["in"] = _graph(case, seed, bases=kind == "step")
        torch.cuda.synchronize()
        s["g"] = cg.cg_load_graph(ctx, s["in"], flags=cg.BORROW_DEVICE | (0 if kind == "step" else cg.NO_READS),
                                  min_chain_reads=case.get("min_chain", 2))
    if kind == "step":
        room = _room(case)
        _fits(cg.cg_emit_contigs(s["g"]), room)
        s["off"] = _zeros(room[0], torch.int64)
        s["bases"] = _zeros(cg.packed_bytes_2bit(room[1]) if case["out"] == "2bit" else room[1])
    elif kind == "reads":
        n = s["g"].n
        s["out"] = [_zeros(n), _zeros(n, torch.int32), _zeros(n, torch.int32), _zeros(n)]
    elif kind == "partition":
        room = _room(case)
        _fits(cg.cg_emit_contigs(s["g"]), room)
        s["part"], s["load"] = _zeros(room[0], torch.int32), _zeros(case["parts"], torch.int64)
    elif kind == "batch":
        sizes = _sizes(case)
        graphs = [_graph(case, seed * 1000 + j, genome) for j, genome in enumerate(sizes)]
        torch.cuda.synchronize()
        s["g"] = cg.cg_load_batch(ctx, graphs)
        room = [sum(r) for r in zip(*(_room(case, genome) for genome in sizes))]
        _fits(cg.cg_emit_contigs(s["g"]), room)
        s["off"], s["bases"] = _zeros(room[0], torch.int64), _zeros(room[1])
        s["ranges"] = [_zeros(case["graphs"] + 1, torch.int64) for _ in range(2)]
    elif kind == "request":
        room = _room(case)
        s["in"] = _to_host(_graph(case, seed))
        s["off"] = _zeros(room[0], torch.int64, pin_memory=True).numpy()
        s["bases"] = _zeros(room[1], pin_memory=True).numpy()
    elif kind == "serve":
        sizes = _sizes(case)
        s["in"] = [_to_host(_graph(case, seed * 1000 + j, genome)) for j, genome in enumerate(sizes)]
        s["room"] = [_room(case, genome) for genome in sizes]
        s["off"] = np.zeros(sum(r[0] for r in s["room"]), dtype=np.int64)
        s["bases"] = np.zeros(sum(r[1] for r in s["room"]), dtype=np.uint8)
        _server()
    elif kind == "reduce":
        s["in"] = d = _graph({**case, "row_bytes": 8}, seed, full=True, bases=False)
        n, m = d.len.numel(), d.col.numel()
        s["desc"] = cg.GraphDesc(n_reads=n, n_entries=m, row_ptr=d.row_ptr.data_ptr(), row_ptr_bytes=8,
                                 mem=cg.MEM_DEVICE, col=d.col.data_ptr(), code=d.code.data_ptr(),
                                 suf=d.suf.data_ptr(), len=d.len.data_ptr())
        m = s["room"] = _reads(case)                  # a third of the reads with two entries, and what repeats add
        s["rows"] = _zeros(n + 1, torch.int64)
        s["out"] = [_zeros(m, torch.int32), _zeros(m), _zeros(m, torch.int32)]
    elif kind == "exchange":
        d = _graph(case, seed)
        n, ranks, room = d.len.numel(), case["ranks"], _room(case)
        rank = s["rank"] = seed % ranks
        s["first"] = first = np.array([n * i // ranks for i in range(ranks + 1)], dtype=np.int64)
        s["in"] = SimpleNamespace(**{**vars(d), "packed": None})
        torch.cuda.synchronize()
        s["g"] = g = cg.cg_load_graph(ctx, s["in"], flags=cg.BORROW_DEVICE | cg.NO_READS)
        _fits(cg.cg_emit_contigs(g), room)
        got = []
        for i in range(ranks):                  # what every rank holds and sends; this rank's own stays in hand
            b0, b1 = int(d.off[first[i]]), int(d.off[first[i + 1]]) if i + 1 < ranks else 4 * d.packed_bytes
            mine, off = d.packed[b0 // 4:b1 // 4].clone(), d.off[first[i]:first[i + 1]] - b0
            buf = _zeros(room[1] // ranks + 8_000_000)
            torch.cuda.synchronize()
            send, _ = cg.cg_exchange_sizes(g, ranks, first, i)
            cg.cg_exchange_pack(g, ranks, first, i, mine, off, buf)
            got.append(buf[send[:rank].sum():send[:rank + 1].sum()])
            if i == rank:
                s["packed"], s["offsets"], s["send"] = mine, off, buf
        s["recv"] = torch.cat(got)
        s["off"], s["share"] = _zeros(room[0], torch.int64), _zeros(room[1] // ranks + 16384)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _spell(g, off, bases, packed=False):
    cg.cg_mask_branches(g, want_count=False)
    cg.cg_chains(g, want_counts=False)
    if packed:
        cg.cg_emit_contigs_2bit(g, off, bases, want_counts=False)
    else:
        cg.cg_emit_contigs(g, off, bases, want_counts=False)


def _serve(s):
    """Submits every request, then takes each result into the program's own buffers."""
    server, lib = _server(), cg.lib()
    ids = [server.submit(g) for g in s["in"]]
    o = b = 0
    for i, room in zip(ids, s["room"]):
        r = cg.ServerResult()
        status = lib.cg_server_wait(server.ptr, i, -1, ctypes.byref(r)) or r.status
        if status != cg.CG_OK:
            raise RuntimeError("a request failed: " + cg.cg_status_str(status))
        _fits((r.n_contigs, r.total_bases), room)
        s["off"][o:o + r.n_contigs + 1] = np.ctypeslib.as_array(r.contig_off, shape=(r.n_contigs + 1,))
        s["bases"][b:b + r.total_bases] = np.ctypeslib.as_array(r.bases, shape=(r.total_bases,))
        server.release(i)
        o, b = o + room[0], b + room[1]
    return [s["off"], s["bases"]]


def run(s):
    case, ctx = s["case"], _context()
    kind = case["kind"]
    if kind == "step":
        _spell(s["g"], s["off"], s["bases"], case["out"] == "2bit")
        return [s["off"], s["bases"]]
    if kind == "reads":
        branch, chain, rank, orient = s["out"]
        cg.cg_mask_branches(s["g"], branch, want_count=False)
        cg.cg_chains(s["g"], chain, rank, orient, want_counts=False)
        return s["out"]
    if kind == "batch":
        _spell(s["g"], s["off"], s["bases"])
        cg.cg_batch_ranges(s["g"], *s["ranges"])
        return [s["off"], s["bases"], *s["ranges"]]
    if kind == "request":
        g = cg.cg_load_graph(ctx, s["in"], flags=cg.HOST_READS)
        _spell(g, s["off"], s["bases"])
        g.close()
        return [s["off"], s["bases"]]
    if kind == "serve":
        return _serve(s)
    if kind == "reduce":
        # the C call with buffers that the program has sized: the reduced graph in one call
        kept = ctypes.c_int64()
        col, code, suf = s["out"]
        status = cg.lib().cg_transitive_reduction(ctx.ptr, ctypes.byref(s["desc"]), 0, s["rows"].data_ptr(),
                                                  col.data_ptr(), code.data_ptr(), suf.data_ptr(), s["room"],
                                                  cg.MEM_DEVICE, ctypes.byref(kept))
        if status != cg.CG_OK:
            raise RuntimeError("the reduction failed: " + cg.cg_status_str(status))
        return [kept.value, s["rows"], *s["out"]]
    if kind == "partition":
        cg.cg_partition_contigs(s["g"], case["parts"], case["weight"], s["part"], s["load"])
        return [s["part"], s["load"]]
    ranks, rank, g = case["ranks"], s["rank"], s["g"]
    send, recv = cg.cg_exchange_sizes(g, ranks, s["first"], rank)
    cg.cg_exchange_pack(g, ranks, s["first"], rank, s["packed"], s["offsets"], s["send"])
    cg.cg_emit_share_received(g, ranks, s["first"], rank, s["recv"], s["off"], s["share"])
    return [send, recv, s["send"], s["off"], s["share"]]


# ------------------------------------------------------- bounds and tolerance
def work(case):
    """Bytes of one pass, from the shape of a graph of the case's distributions: 8 or 4 bytes of row offset per
    read, 9 per overlap entry, 12 per spelled read, a quarter byte read and one (2-bit: a quarter) written per
    contig base, contig bases about the genome's."""
    kind = case["kind"]
    genomes = _sizes(case) if "graphs" in case else [case["genome"]]
    total = 0
    for genome in genomes:
        n = _reads(case, genome)
        kept = min(n, 2.0 * genome / case["mean"])               # uncontained reads: about two per mean length
        rows, entries, spelled = n * case.get("row_bytes", 4), 9 * 2 * kept, 12 * kept
        bases = genome * (case["coverage"] if case.get("min_chain") == 1 else 1)
        if kind == "step":
            total += rows + entries + spelled + bases * (0.5 if case["out"] == "2bit" else 1.25)
        elif kind == "reads":
            total += rows + entries + 10 * n
        elif kind == "reduce":
            total += n * (8 + 4 + 8) + 9 * 8 * kept + 9 * 2 * kept    # full rows of about eight, two kept
        elif kind == "partition":
            total += 2.3e-6 * 2 * genome * 12 + 8 * case["parts"]
        elif kind == "exchange":
            total += rows + entries + spelled + bases / case["ranks"] * (0.25 + 0.25 + 0.25 + 1)
        elif kind == "batch":
            total += 2 * rows + entries + spelled + bases * 1.25
        else:                                                      # from and to host memory
            total += n * (4 + 12) + entries + spelled + bases * 1.25
    return {"bytes": total, "flops": 0}


def tolerance(case):
    return "exact"
