"""The benchmark's recorded DRAM traffic is tied to the sources that decide it: the
ASCII spelling kernel and the plan of its spans."""
import os
import shutil

import bench

CSRC = os.path.join(bench.ROOT, "paper_2207_04350_gb300", "csrc")


def test_a_change_of_either_source_changes_the_fingerprint(tmp_path):
    for name in bench.EMIT_SOURCES:
        shutil.copy(os.path.join(CSRC, name), tmp_path)
    assert bench.emit_source_sha256_16(str(tmp_path)) == bench.emit_source_sha256_16()
    for name in bench.EMIT_SOURCES:
        text = (tmp_path / name).read_bytes()
        (tmp_path / name).write_bytes(text + b"\n")
        assert bench.emit_source_sha256_16(str(tmp_path)) != bench.emit_source_sha256_16()
        (tmp_path / name).write_bytes(text)


def test_the_sources_hold_the_kernel_and_its_plan():
    text = "".join(open(os.path.join(CSRC, name)).read() for name in bench.EMIT_SOURCES)
    for what in ("k_emit(Scratch s", "struct SpanPlan {", "inline int emit_span(", "struct TileQueue {"):
        assert what in text, what
