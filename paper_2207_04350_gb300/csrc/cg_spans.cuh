// cg_spans.cuh - how a spelling launch cuts its output tiles into spans and hands
// them to its warps (sm_103a). With cg_emit.cu this is what the DRAM traffic of the
// ASCII spelling depends on: the benchmark's recorded figure is tied to both files.
#pragma once

#include <cuda_runtime.h>

namespace cg {

// Output tiles [t_begin, t_stop) for the W warps of a persistent grid: warp gw
// spells tile t_begin + gw first; the tiles from t_begin + W on go out one at a
// time, the tiles t_begin + W + c + kTicketSets * k from counter c (zeroed
// before the launch) to the warps gw = c mod kTicketSets, each warp asking for
// its next ticket while it spells its current tile. A warp thus takes its next
// tile when it finishes one, and the warps end together whatever each tile
// holds; no launch starts with every warp on one counter, and a launch with no
// more tiles than warps touches no counter.
constexpr int kTicketSets = 8, kTicketStride = 16;

struct TileQueue {
  long long t;                 // the warp's current tile (past t_stop: done)
  unsigned long long tk;
  __device__ static long long warp_id() {
    return (long long)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  }
  __device__ static long long warps() { return (long long)gridDim.x * (blockDim.x >> 5); }
  __device__ TileQueue(long long t_begin) : t(t_begin + warp_id()), tk(0) {}
  // The warp's current tile is t while t < t_stop; call ask() as the tile is
  // started and next() when it is done (warp-uniform calls, with the launch's
  // counters and tile range; the queue keeps no copy, to spare registers). A
  // grid with no fewer warps than tiles takes no ticket.
  __device__ void ask(unsigned long long* tickets, long long t_begin, long long t_stop, int lane) {
    if (t_begin + warps() < t_stop && lane == 0)
      tk = atomicAdd(tickets + kTicketStride * (int)(warp_id() % kTicketSets), 1ull);
  }
  __device__ void next(long long t_begin, long long t_stop) {
    const long long k = (long long)__shfl_sync(0xffffffffu, tk, 0);
    t = t_begin + warps() < t_stop ? t_begin + warps() + warp_id() % kTicketSets + (long long)kTicketSets * k
                                   : 0x7fffffffffffffffll;
  }
};

// Layout tiles a spelling warp takes at once: emit_tile / layout tile when the
// caller set one (at least one tile), else the largest span of at most max_bytes
// that leaves every one of the launch's warps at least per_warp spans of the n
// layout tiles (big outputs: big spans, few per-span overheads; small ones: one
// layout tile, enough spans to balance). The 2-bit kernel, whose fixed cost per
// span weighs four times more against its bytes, asks for 2 per warp of at most
// 32 KiB.
__host__ __device__ inline int emit_span(long long n_tiles, long long warps, int emit_tile, int layout_tile,
                                         int per_warp, int max_bytes) {
  if (emit_tile > 0) return emit_tile > layout_tile ? emit_tile / layout_tile : 1;
  int span = 1;
  while (2 * span * layout_tile <= max_bytes && n_tiles / (2 * span) >= per_warp * warps) span *= 2;
  return span;
}

// The ASCII kernel's spans: of layout tiles [t0, t1), as many of emit_span's size
// (8 per warp, at most 64 KiB) as leave one per warp, and the rest in eighths of it
// (of 8 KiB at least), so that the warps end together although the spans are big.
// Against spans of one size of at most 32 KiB, k_emit on 3.1 Gb: 679 to 671 us;
// whole steps: 3.1 Gb 830 to 822 us, 1.3 Gb 404 to 399. At most 128 KiB gave no more; 4 per warp made steps of 500 Mb 2% faster and
// 1.2 Gb of lone reads 2.5% slower (288 to 294 us); halves at the end gave a third
// of it. The 2-bit kernel keeps one size: 141.3 us on 1.2 Gb with or without halves
// at the end, 145.4 with quarters.
struct SpanPlan {
  long long t0, t1, big;       // big: how many spans of the full size
  int span, small;
  __device__ SpanPlan(long long t_begin, long long t_stop, long long warps, int emit_tile, int layout_tile)
      : t0(t_begin), t1(max(t_begin, t_stop)) {
    span = emit_span(t1 - t0, warps, emit_tile, layout_tile, 8, 65536);
    small = emit_tile > 0 ? span : min(span, max(span / 8, 8192 / layout_tile));
    big = small == span ? 0 : max(0ll, (t1 - t0) / span - warps);
  }
  __device__ long long spans() const { return big + (t1 - t0 - big * span + small - 1) / small; }
  __device__ long long first(long long i) const {        // first tile of span i; t1 past the last
    return min(t1, t0 + (i < big ? i * span : big * span + (i - big) * small));
  }
};

}  // namespace cg
