"""Failure handling with host-side fault injection (no GPU fault, trap or
hang): each injected failure is reported with its status; CG_ECUDA,
CG_ETIMEOUT and CG_EKERNEL make the context refuse further work until it is
destroyed, CG_ENOMEM and CG_EGRAPH do not; a fresh context (or the same one,
for the recoverable ones) then gives bit-exact results. Server: admission
refusals and a stalled worker (a bounded wait gives up, the request still
completes). One device wait really runs out: the look-back scan with its
first tile withheld returns by itself with CG_ETIMEOUT."""
import os

import numpy as np
import pytest

import gen
import oracle
from paper_2207_04350_gb300 import cg
from tests._exchange import without_reads
from tests._graphs import structured

torch = pytest.importorskip("torch")
I32, I64 = torch.int32, torch.int64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiny():
    import torch
    from paper_2207_04350_gb300 import _build
    _build.build()
    assert torch.cuda.is_available()
    G = gen.generate("tiny-1Mb", threads=8)
    return G, oracle.run(G, min_chain_reads=2)


def contigs(ctx, G):
    g = cg.cg_load_graph(ctx, G)
    try:
        return cg.contigs_host(g)
    finally:
        g.close()


def exact(ctx, G, orc):
    off, bases = contigs(ctx, G)
    assert np.array_equal(off, orc.contig_off) and np.array_equal(bases, orc.bases)


def test_device_wait_runs_out(tiny):
    """A real device-side wait that runs out, not an injected status: the
    look-back scan with tile 0 withheld, so the later tiles wait on a
    descriptor that nothing publishes until their bounded wait gives up. The
    kernel returns by itself with CG_ETIMEOUT recorded; the context then
    refuses work, and a fresh context on the same GPU is bit-exact."""
    import time
    G, orc = tiny
    ctx = cg.cg_create(0)
    try:
        exact(ctx, G, orc)
        t0 = time.perf_counter()
        st = cg.cg_selftest_wait_timeout(ctx, 4)
        waited = time.perf_counter() - t0
        assert st == cg.CG_ETIMEOUT, cg.cg_status_str(st)
        assert waited < 30.0
        for call in (lambda: cg.cg_sync(ctx), lambda: contigs(ctx, G)):
            with pytest.raises(cg.CgError) as e:
                call()
            assert e.value.status == cg.CG_ETIMEOUT
    finally:
        ctx.close()
    ctx = cg.cg_create(0)
    try:
        exact(ctx, G, orc)
    finally:
        ctx.close()


@pytest.mark.parametrize("site,at,status,sticky", [
    ("alloc", 3, cg.CG_ENOMEM, False),
    ("bad_graph", 1, cg.CG_EGRAPH, False),
    ("h2d", 2, cg.CG_ECUDA, True),
    ("timeout", 2, cg.CG_ETIMEOUT, True),
    ("kernel", 1, cg.CG_EKERNEL, True),
])
def test_injected_failure(tiny, site, at, status, sticky):
    G, orc = tiny
    ctx = cg.cg_create(0)
    try:
        cg.cg_set_fault(ctx, f"{site}:{at}")
        with pytest.raises(cg.CgError) as e:
            contigs(ctx, G)
        assert e.value.status == status
        if sticky:
            with pytest.raises(cg.CgError) as e2:
                contigs(ctx, G)
            assert e2.value.status == status
        else:
            exact(ctx, G, orc)                   # the same context goes on
    finally:
        ctx.close()
    fresh = cg.cg_create(0)
    try:
        exact(fresh, G, orc)
    finally:
        fresh.close()


# What each call that writes outputs is given: the load's flags, then the outputs' sizes
# in bytes from (reads, contigs, bases), then the call.
AFTER_A_TIMEOUT = {
    "contigs": (0, lambda n, c, b: (8 * (c + 1), b + 16),
                lambda g, o: cg.cg_emit_contigs(g, o[0].view(I64), o[1], want_counts=False)),
    "contigs-after-chains": (0, lambda n, c, b: (8 * (c + 1), b + 16),
                             lambda g, o: (cg.cg_chains(g, want_counts=False),
                                           cg.cg_emit_contigs(g, o[0].view(I64), o[1], want_counts=False))),
    "offsets": (0, lambda n, c, b: (8 * (c + 1),),
                lambda g, o: cg.cg_emit_contigs(g, o[0].view(I64), None, want_counts=False)),
    "2bit": (0, lambda n, c, b: (8 * (c + 1), 16 * (b // 64 + 1)),
             lambda g, o: cg.cg_emit_contigs_2bit(g, o[0].view(I64), o[1], want_counts=False)),
    "share": (0, lambda n, c, b: (8 * (c + 1), b + 16),
              lambda g, o: cg.cg_emit_share(g, 0, 2, o[0].view(I64), o[1], want_range=False)),
    "reads": (0, lambda n, c, b: (4 * n, 4 * n, n),
              lambda g, o: cg.cg_chains(g, o[0].view(I32), o[1].view(I32), o[2], want_counts=False)),
    "part": (0, lambda n, c, b: (4 * c, 8 * 24),
             lambda g, o: cg.cg_partition_contigs(g, 24, part=o[0].view(I32), part_weight=o[1].view(I64))),
    "exchange": (cg.NO_READS, lambda n, c, b: (), lambda g, o: cg.cg_exchange_sizes(g, 2, [0, g.n // 2, g.n], 0)),
}


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("call", list(AFTER_A_TIMEOUT))
def test_nothing_runs_on_after_a_wait_that_gave_up(tiny, call, graphs):
    """A grid barrier that gave up leaves contig records unwritten, which the later
    kernels would use as indices: with the error word as it leaves it, on a graph with
    a chain long enough for the barrier and with closed chains, no output is written,
    the next wait reports CG_ETIMEOUT and a fresh context is bit-exact."""
    flags, sizes, run = AFTER_A_TIMEOUT[call]
    G = structured(23, [30] * 800 + [6000] + [900] * 3, closed=[False] * 801 + [True] * 3)
    orc = oracle.run(G, min_chain_reads=2)
    out = [torch.full((b,), 0xA5, dtype=torch.uint8, device="cuda")
           for b in sizes(G.n, len(orc.contig_off) - 1, len(orc.bases))]
    ctx = cg.cg_create(0)
    try:
        cg.cg_set_graphs(ctx, graphs)
        g = cg.cg_load_graph(ctx, without_reads(G) if flags & cg.NO_READS else G, flags=flags, min_chain_reads=2)
        cg.cg_set_fault(ctx, "barrier:1")
        with pytest.raises(cg.CgError) as e:
            run(g, out)
            cg.cg_sync(ctx)
        assert e.value.status == cg.CG_ETIMEOUT
        assert all(bool((t == 0xA5).all()) for t in out)
        g.close()
    finally:
        ctx.close()
    fresh = cg.cg_create(0)
    try:
        exact(fresh, G, orc)
    finally:
        fresh.close()


def test_a_stage_is_captured_when_it_comes_twice_in_a_row(tiny):
    """Two output buffers used in turn are no reason to capture again: the first keeps
    its graph and the other is launched, until one comes twice in a row."""
    G, orc = tiny
    out = [torch.zeros(len(orc.bases) + 16, dtype=torch.uint8, device="cuda") for _ in range(2)]
    off = torch.zeros(len(orc.contig_off), dtype=I64, device="cuda")
    ctx = cg.cg_create(0)
    try:
        g = cg.cg_load_graph(ctx, G)

        def step(k):
            out[k].zero_()
            torch.cuda.synchronize()
            cg.cg_mask_branches(g, want_count=False)
            cg.cg_chains(g, want_counts=False)
            cg.cg_emit_contigs(g, off, out[k], want_counts=False)
            cg.cg_sync(ctx)
            assert np.array_equal(out[k][:len(orc.bases)].cpu().numpy(), orc.bases)

        step(0)
        step(0)                                  # captured
        cg.cg_set_fault(ctx, "capture:1")
        for k in (1, 0, 1, 0, 0, 1, 0, 1):
            step(k)
        with pytest.raises(cg.CgError) as e:
            step(1)                              # twice in a row: captured, which the plan fails
        assert e.value.status == cg.CG_ECUDA
        g.close()
    finally:
        ctx.close()


def test_plan_from_environment(tiny):
    G, orc = tiny
    os.environ["CG_FAULT"] = "bad_graph:2"
    try:
        ctx = cg.cg_create(0)
    finally:
        del os.environ["CG_FAULT"]
    try:
        exact(ctx, G, orc)                       # the first load passes
        with pytest.raises(cg.CgError) as e:
            contigs(ctx, G)
        assert e.value.status == cg.CG_EGRAPH
        exact(ctx, G, orc)
        cg.cg_set_fault(ctx, None)
    finally:
        ctx.close()


def server_with(plan, **kw):
    os.environ["CG_FAULT"] = plan
    try:
        return cg.Server(0, **kw)
    finally:
        del os.environ["CG_FAULT"]


def check_result(res, orc):
    assert res["status"] == cg.CG_OK
    assert np.array_equal(res["contig_off"], orc.contig_off) and np.array_equal(res["bases"], orc.bases)


def test_server_admission_refused(tiny):
    G, orc = tiny
    srv = server_with("admit:2", hbm_budget_bytes=8 << 30, max_batch=4, workers=2)
    try:
        a = srv.submit(G)
        with pytest.raises(cg.CgError) as e:
            srv.submit(G)
        assert e.value.status == cg.CG_EBUSY
        b = srv.submit(G)
        for rid in (a, b):
            check_result(srv.wait(rid), orc)
            srv.release(rid)
    finally:
        srv.stop()


def test_server_worker_stall(tiny):
    G, orc = tiny
    srv = server_with("queue_stall:1:600", hbm_budget_bytes=8 << 30, max_batch=4, workers=1)
    try:
        rid = srv.submit(G)
        with pytest.raises(cg.CgError) as e:
            srv.wait(rid, timeout_ms=50)          # the worker is stalled: the bounded wait gives up
        assert e.value.status == cg.CG_ETIMEOUT
        check_result(srv.wait(rid), orc)         # and the request still completes
        srv.release(rid)
    finally:
        srv.stop()


def test_server_replaces_a_refusing_context(tiny):
    """A batch whose device wait reports a timeout leaves its context refusing
    work; the worker replaces that context, so the failed batch's request
    reports CG_ETIMEOUT and every later request is bit-exact."""
    G, orc = tiny
    srv = server_with("batch_timeout:1", hbm_budget_bytes=8 << 30, max_batch=4, workers=1)
    try:
        rid = srv.submit(G)
        res = srv.wait(rid)
        assert res["status"] == cg.CG_ETIMEOUT
        srv.release(rid)
        for _ in range(3):
            rid = srv.submit(G)
            check_result(srv.wait(rid), orc)
            srv.release(rid)
        assert srv.stats()["contexts_replaced"] == 1
    finally:
        srv.stop()


def test_server_malformed_request_fails_alone(tiny):
    """One malformed graph batched with valid ones: the union fails its input
    checks, the batch is run again one request at a time, and only the
    malformed request reports CG_EGRAPH; the others are bit-exact."""
    G, orc = tiny
    B = type("B", (), {})()
    for k in ("row_ptr", "col", "code", "suf", "len", "off", "packed"):
        setattr(B, k, np.array(getattr(G, k), copy=True))
    B.code[0] ^= 1                                # the entry no longer matches its mirror
    assert not oracle.validate(B)[0]
    # the first batch stalls, so the requests submitted meanwhile form one batch
    srv = server_with("queue_stall:1:500", hbm_budget_bytes=8 << 30, max_batch=16, workers=1)
    try:
        first = srv.submit(G)
        ids = [(srv.submit(B if i == 2 else G), i == 2) for i in range(5)]
        check_result(srv.wait(first), orc)
        srv.release(first)
        for rid, bad in ids:
            res = srv.wait(rid)
            if bad:
                assert res["status"] == cg.CG_EGRAPH
            else:
                check_result(res, orc)
            srv.release(rid)
        assert srv.stats()["batches"] == 2       # the five shared one batch
    finally:
        srv.stop()
