// cg_scan.cu - output layout of the contigs (sm_103a): the single-GPU form of
// the contig-size estimate, the redistribution by contig and the offsets of
// the concatenation (Alg. 2, Sec. 4.2-4.4).
//
//   1. scan over the words of the heads bitmap (bit m set when read m is the
//      smallest read of a contig) of their heads and those heads' read
//      counts: the contig index of every head, listing contigs by smallest
//      read id, and every contig's first walk position and read count;
//   2. scatter every spelled read to walk position first(contig) + rank: the
//      on-device compaction that replaces the induced-subgraph exchange;
//   3. scan over walk positions of the bases each read adds: the output
//      offset of every piece, the contig offsets and the map from output
//      tiles to the piece holding each tile's first byte.
//
// For one part of a contig partition (cg_emit_part, Sec. 4.3) step 2 gives
// the reads of other parts' contigs empty pieces, so step 3 lays out that
// part's contigs alone, back to back.
//
// The scan of step 1 takes a block per tile, and whoever marks a head also adds
// it to the sum of its tile (mark_head, and the mask's lone reads): a tile's
// start is the sum of the tile sums before it, read by its own block, and no
// block waits for another. There are at most 2048 tiles; larger graphs have
// larger ones. The scan of step 3 is a single-pass decoupled look-back scan
// (cg_lookback.cuh), whose wait on a predecessor is bounded.
#include <cuda_runtime.h>

#include <algorithm>

#include "cg_internal.cuh"
#include "cg_lookback.cuh"

namespace cg {

namespace {

// Block-wide exclusive prefix of one 64-bit value per thread; the sum of all in
// *total. `tot` is shared memory of kBlock / 32 words, free again after a barrier.
__device__ __forceinline__ unsigned long long block_exclusive(unsigned long long v, unsigned long long* tot,
                                                              unsigned long long* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) tot[warp] = inc;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kBlock / 32; ++w) {
    if (w < warp) before += tot[w];
    all += tot[w];
  }
  *total = all;
  return before + inc - v;
}

// Block-wide sum, the same scratch.
__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long* tot) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) tot[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long all = 0;
#pragma unroll
  for (int w = 0; w < kBlock / 32; ++w) all += tot[w];
  return all;
}

// Contig index and first walk position of every head, a block per tile of the
// heads bitmap (256 words or more). The value of a word packs the contigs
// headed in it (their count, above bit kHeadShift) and their reads (below):
// both stay under 2^30, so one scan gives every head its contig index and its
// contig's first walk position at once. A lone read's contig has one read; only
// the chain heads' read counts are loaded. The kernels that marked the heads
// added up every tile's sum (hsum), so a block adds the sums before its tile,
// a load or a few per thread, and waits for no other block: what bounds it is
// three dependent loads and the block scan: 14.3 us by events on the 3.1 Gb
// graph. With tiles of 2048 words that looked back over their predecessors it
// took 30.7 us there (95 tiles in flight at once, each waiting for the one
// before), and 131 us on 94 thousand lone reads, whose 32 heads per word one
// thread then loaded in turn (the whole step: 397 us before, 283 now).
__global__ void __launch_bounds__(kBlock) k_heads(Scratch s, long long n, int64_t* user_off, long long user_cap) {
  pdl_enter();
  __shared__ unsigned long long tot[2][kBlock / 32];   // the prefix's sums, the words' sums
  for (long long i = grid_tid(); i <= s.scan_tiles_cap; i += grid_threads()) s.scan_state[i] = 0ull;   // of the piece scan
  const int tile = (int)blockIdx.x, tid = threadIdx.x;
  unsigned long long run = 0;
  for (int i = tid; i < tile; i += kBlock) run += s.hsum[i];
  const long long per = 1ll << (s.h_shift - 5);
  const long long w_end = min((n + 31) / 32, (tile + 1) * per);
  bool first = true;
  for (long long wb = tile * per; wb < w_end; wb += kBlock) {
    const long long w = wb + tid;
    unsigned bits = w < w_end ? s.hb[w] : 0u;
    const unsigned lone = w < w_end ? s.hb_mask[w] : 0u, chain = bits & ~lone;
    const int32_t* const hq = s.headq + 32 * w;
    const unsigned q0 = chain ? (unsigned)hq[__ffs(chain) - 1] : 0u;
    unsigned long long reads = __popc(lone) + q0;
    for (unsigned c = chain & (chain - 1); c; c &= c - 1) reads += (unsigned)hq[__ffs(c) - 1];   // rare
    if (first) {
      run = block_sum(run, tot[1]);
      first = false;
    }
    unsigned long long all;
    const unsigned long long e =
        run + block_exclusive(((unsigned long long)__popc(bits) << kHeadShift) | reads, tot[0], &all);
    if (w < w_end) {
      unsigned k = (unsigned)(e >> kHeadShift);
      unsigned long long r = e & ((1ull << kHeadShift) - 1);
      s.wp[w] = k;
      for (; bits; bits &= bits - 1, ++k) {            // contigs in order of their smallest read
        const int b = __ffs(bits) - 1;
        const unsigned q = (lone >> b) & 1u ? 1u : (b == __ffs(chain) - 1 ? q0 : (unsigned)hq[b]);
        s.qd[k] = (int32_t)q;
        s.cbase[k] = r;
        r += q;
      }
    }
    run += all;
    __syncthreads();                                   // tot is reused by the next words
  }
  if (tile == (int)gridDim.x - 1 && tid == 0) {
    Counters* c = s.ctr;
    unsigned C = (unsigned)(run >> kHeadShift);
    unsigned long long W = run & ((1ull << kHeadShift) - 1);
    if (W > (unsigned long long)n) {                   // contigs of more reads than there are: not a string graph
      set_error(s.derr, DERR_KERNEL, K_SCAN_HEADS, (long long)W);
      C = 0;
      W = 0;
    }
    c->n_contigs = C;
    s.cbase[C] = W;
    c->n_walk = (unsigned)W;
    if (C == 0) {                                      // no contigs: the piece scan has nothing to scan
      s.contig_off[0] = 0;
      if (user_off && user_cap >= 1) user_off[0] = 0;
      c->total_bases = 0;
      c->n_tiles = 0;
    }
  }
}

// What the piece scan writes for walk position j: a piece of L bases from
// output offset o on, the first of contig `starts` (or -1).
struct PieceStore {
  int64_t* out_off;
  int64_t* contig_off;
  int32_t* tile_seg;
  long long tiles_cap;
  long long tile_bytes;
  Counters* c;
  DevError* derr;
  // The caller's contig offsets, when the offsets are spelled for a caller
  // buffer in the same replayed stage: written here instead of by a copy kernel
  // afterwards, and only when all n_contigs + 1 fit (else a capacity error).
  int64_t* user_off;
  long long user_cap;
  __device__ bool user_fits() const {
    return user_off && (long long)*(const volatile unsigned*)&c->n_contigs + 1 <= user_cap;
  }
  __device__ void item(long long j, long long o, long long L, int32_t starts) const {
    out_off[j] = o;
    if (starts >= 0) {
      contig_off[starts] = o;
      if (user_fits()) user_off[starts] = o;
    }
    // tile_bytes is a power of two: the first tile starting at or after o, and after o + L
    const int sh = __ffsll(tile_bytes) - 1;
    long long t0 = (o + tile_bytes - 1) >> sh, t1 = (o + L + tile_bytes - 1) >> sh;
    for (long long t = t0; t < t1; ++t) {
      if (t < tiles_cap) tile_seg[t] = (int32_t)j;
      else set_error(derr, DERR_KERNEL, K_SCAN_OFFSETS, t);
    }
  }
  __device__ void last(long long count, unsigned long long total) const {
    out_off[count] = (long long)total;
    contig_off[c->n_contigs] = (long long)total;
    if (user_off) {
      if (user_fits()) user_off[c->n_contigs] = (long long)total;
      else set_error(derr, DERR_CAPACITY, K_CONTIG_OFF, (long long)c->n_contigs + 1);
    }
    c->total_bases = (long long)total;
    long long nt = ((long long)total + tile_bytes - 1) / tile_bytes;
    c->n_tiles = (unsigned)nt;
    if (nt <= tiles_cap) tile_seg[nt] = (int32_t)(count - 1);
    else set_error(derr, DERR_KERNEL, K_SCAN_OFFSETS, nt);
  }
};

// Piece offsets over the walk positions, in tiles of kPieceTile positions, four
// per thread, with a decoupled look-back (cg_lookback.cuh). Adding up every
// tile's bases in the scatter instead, as the heads' sums are, cost the scatter
// 30 us on the 3.1 Gb graph (a thousand additions to each of 410 words).
constexpr int kPieceItems = kPieceTile / kBlock;
static_assert(kPieceItems == 4, "one 16-byte load per thread and array");

__global__ void __launch_bounds__(kBlock) k_pieces(Scratch s, PieceStore ps) {
  pdl_enter();
  __shared__ unsigned long long tot[kBlock / 32];
  __shared__ long long s_tile;
  const int tid = threadIdx.x;
  const long long W = *(const volatile unsigned*)&s.ctr->n_walk;
  const long long tiles = (W + kPieceTile - 1) / kPieceTile;
  if (blockIdx.x == 0 && tid < kTicketSets) s.tickets[kTicketStride * tid] = 0ull;   // for a spelling right after
  if ((long long)blockIdx.x >= tiles) return;
  for (;;) {
    if (tid == 0) s_tile = (long long)atomicAdd(&s.scan_state[s.scan_tiles_cap], 1ull);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= tiles) return;                         // block-uniform
    const long long i0 = tile * kPieceTile + kPieceItems * tid;
    int32_t L[kPieceItems], f[kPieceItems];
    if (i0 + kPieceItems <= W) {
      const int4 a = *reinterpret_cast<const int4*>(s.wlen + i0), b = *reinterpret_cast<const int4*>(s.wfirst + i0);
      L[0] = a.x; L[1] = a.y; L[2] = a.z; L[3] = a.w;
      f[0] = b.x; f[1] = b.y; f[2] = b.z; f[3] = b.w;
    } else {
#pragma unroll
      for (int k = 0; k < kPieceItems; ++k) {
        L[k] = i0 + k < W ? s.wlen[i0 + k] : 0;
        f[k] = i0 + k < W ? s.wfirst[i0 + k] : -1;
      }
    }
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < kPieceItems; ++k) sum += (unsigned)L[k];
    unsigned long long all, e = block_exclusive(sum, tot, &all);
    e += lookback(s.scan_state, tile, all, s.derr, (int)K_SCAN_OFFSETS);
#pragma unroll
    for (int k = 0; k < kPieceItems; ++k) {
      if (i0 + k >= W) break;
      ps.item(i0 + k, (long long)e, L[k], f[k]);
      e += (unsigned)L[k];
      if (i0 + k == W - 1) ps.last(W, e);
    }
    __syncthreads();                                   // s_tile and tot are reused by the next tile
  }
}

// Every spelled read goes to walk position first(contig) + rank, with the
// stored-base address of its piece (for one part's layout, an empty piece
// when its contig belongs to another part): forward reads add stored bases
// [len-contrib, len), reverse-complement reads the complement of stored
// bases contrib-1 down to 0. The spelled reads are the lone reads of the mask
// stage (each its own contig, whole and forward) and the candidates with a
// contig in their record (chains long enough, and reads cut off by branch
// reads when those are spelled alone). A thread takes two reads at a time and
// issues each level of their dependent loads together, before any store.
constexpr int kScatterItems = 2;

__global__ void k_scatter(DevGraph g, Scratch s) {
  pdl_enter();
  Counters* c = s.ctr;
  const long long L1 = *(volatile unsigned*)&c->n_lone, NC = *(volatile unsigned*)&c->n_cand;
  const long long W = *(volatile unsigned*)&c->n_walk;
  const long long total = L1 + NC;
  const long long T = grid_threads();
  for (long long k0 = grid_tid(); k0 < total; k0 += kScatterItems * T) {
    long long k[kScatterItems];
    int32_t v[kScatterItems];
    int4 p[kScatterItems];
    bool ok[kScatterItems];
#pragma unroll
    for (int j = 0; j < kScatterItems; ++j) {
      k[j] = k0 + j * T;
      v[j] = k[j] >= total ? 0 : (k[j] < L1 ? s.lone[k[j]] : s.cand[k[j] - L1]);
      // a lone read: its own contig, rank 0, whole and forward (its length is filled in below)
      p[j] = k[j] >= total ? make_int4(-1, 0, 0, 0) : (k[j] < L1 ? make_int4(v[j], 0, -1, 0) : s.prd[k[j] - L1]);
      ok[j] = p[j].x >= 0;                 // not a chain shorter than min_chain
    }
    unsigned word[kScatterItems], wpv[kScatterItems];
    int32_t L[kScatterItems], pf[kScatterItems];
    int64_t base[kScatterItems];
#pragma unroll
    for (int j = 0; j < kScatterItems; ++j) {
      const int32_t m = ok[j] ? p[j].x : 0;
      word[j] = ok[j] ? s.hb[m >> 5] : 0u;
      wpv[j] = ok[j] ? s.wp[m >> 5] : 0u;
      L[j] = ok[j] ? g.len[v[j]] : 0;
      base[j] = ok[j] ? g.off[v[j]] : 0;
      pf[j] = ok[j] && g.pre && k[j] >= L1 ? s.pfirst[k[j] - L1] : 0;
    }
    long long cidx[kScatterItems], pos[kScatterItems];
#pragma unroll
    for (int j = 0; j < kScatterItems; ++j) {
      const int32_t m = p[j].x;
      cidx[j] = (long long)wpv[j] + __popc(word[j] & ((1u << (m & 31)) - 1u));
      pos[j] = ok[j] ? (long long)s.cbase[cidx[j]] + p[j].y : 0;
    }
#pragma unroll
    for (int j = 0; j < kScatterItems; ++j) {
      if (!ok[j]) continue;
      const int32_t m = p[j].x, rk = p[j].y;
      if (!((word[j] >> (m & 31)) & 1u) || pos[j] >= W) { set_error(s.derr, DERR_KERNEL, K_SCATTER, v[j]); continue; }
      const int o = p[j].w;
      const int32_t cb = p[j].z < 0 ? L[j] : p[j].z;
      // stored index of the piece's first base: suffix form, the last cb bases
      // of the oriented read; x-drop form, set by the chain stage (a read spelled
      // alone is whole and forward)
      const int64_t first = !g.pre ? (o == 0 ? L[j] - cb : cb - 1) : pf[j];
      const unsigned long long src = o == 0 ? (unsigned long long)(base[j] + first)
                                            : ((unsigned long long)(base[j] + first) | (1ull << 63));
      s.wsrc[pos[j]] = src;
      s.wlen[pos[j]] = s.part && s.part[cidx[j]] != s.part_p ? 0 : cb;   // another part's contig: empty
      s.wfirst[pos[j]] = rk == 0 ? (int32_t)cidx[j] : -1;
      if (s.wread) s.wread[pos[j]] = v[j];           // a graph without its reads: for the read exchange
    }
  }
}

// An empty graph: no contigs, and the one offset 0.
__global__ void k_contig_off(Scratch s) {
  pdl_enter();
  if (grid_tid() == 0) {
    s.contig_off[0] = 0;
    s.ctr->n_contigs = 0;
    s.ctr->n_walk = 0;
    s.ctr->n_tiles = 0;
    s.ctr->total_bases = 0;
  }
}

__global__ void k_export_contig_off(Scratch s, int64_t* out, long long cap) {
  pdl_enter();
  Counters* c = s.ctr;
  long long C = *(volatile unsigned*)&c->n_contigs;
  if (C + 1 > cap) {
    if (grid_tid() == 0) set_error(s.derr, DERR_CAPACITY, K_CONTIG_OFF, C + 1);
    return;
  }
  for (long long i = grid_tid(); i <= C; i += grid_threads()) out[i] = s.contig_off[i];
}

}  // namespace

cudaError_t launch_offsets(const DevGraph& g, const Scratch& s, const Tuning& t, const LaunchEnv& env,
                           int64_t* user_off, long long user_cap) {
  if (g.n == 0) {
    k_contig_off<<<1, kBlock, 0, env.stream>>>(s);
    mark(env, "k_contig_off");
    return cudaGetLastError();
  }
  cudaError_t e = launch_k(k_heads, s.h_tiles, env, env.pdl_first, s, (long long)g.n, user_off, user_cap);
  if (e != cudaSuccess) return e;
  mark(env, "k_heads");
  static const int scatter_resident = resident_blocks(k_scatter);   // a persistent grid
  const long long scatter_need = (g.n + (long long)kBlock * kScatterItems - 1) / ((long long)kBlock * kScatterItems);
  e = launch_k(k_scatter, (int)std::max(1LL, std::min((long long)env.num_sms * scatter_resident, scatter_need)), env,
               true, g, s);
  if (e != cudaSuccess) return e;
  mark(env, "k_scatter");
  PieceStore ps{s.out_off, s.contig_off, s.tile_seg, s.tiles_cap, t.tile_bytes, s.ctr, s.derr, user_off, user_cap};
  e = launch_k(k_pieces, (int)std::min((long long)s.scan_tiles_cap, (long long)env.num_sms * 4), env, true, s, ps);
  if (e != cudaSuccess) return e;
  mark(env, "k_pieces");
  return cudaGetLastError();
}

namespace {
struct ZeroLoad {
  __device__ unsigned long long operator()(long long) const { return 0ull; }
};
struct NoStore {
  __device__ void item(long long, unsigned long long) const {}
  __device__ void last(long long, unsigned long long) const {}
};
}  // namespace

cudaError_t launch_selftest_wait(unsigned long long* state, long long tiles, DevError* derr, const LaunchEnv& env) {
  k_scan<<<scan_grid(tiles, env), kBlock, 0, env.stream>>>(ZeroLoad{}, NoStore{}, tiles * kTileItems, state,
                                                           tiles, derr, (int)K_SELFTEST_WAIT);
  mark(env, "k_scan_selftest");
  return cudaGetLastError();
}

cudaError_t launch_export_contig_off(const Scratch& s, int64_t* out, int64_t cap, const LaunchEnv& env) {
  cudaError_t e = launch_k(k_export_contig_off, env.num_sms, env, env.pdl_first, s, out, (long long)cap);
  if (e != cudaSuccess) return e;
  mark(env, "k_export_contig_off");
  return cudaGetLastError();
}

}  // namespace cg

// ------------------------------------------------------------------------
// GreedyPartitioning (LPT, Sec. 4.3). Contigs are weighted by their number of
// reads (the size estimate of Sec. 4.3) or by their spelled bases, sorted by
// weight, largest first, equal weights in contig order, and each in turn goes
// to the part whose weight sum is smallest so far, the lowest part on ties.
// The sort is a stable LSD radix sort, 8-bit digits, of kmax - weight; the
// assignment is sequential by definition and runs in one warp.
namespace cg {

namespace {

constexpr int kSortItems = 8;
constexpr long long kSortTile = (long long)kSortItems * kBlock;     // 2048 keys per tile

__device__ __forceinline__ unsigned digit_of(unsigned long long key, int pass) {
  return (unsigned)((key >> (8 * pass)) & 255ull);
}

__global__ void k_sort_keys(const Scratch s, long long C, int weight, unsigned long long kmax, unsigned long long* key,
                            int32_t* val) {
  for (long long i = grid_tid(); i < C; i += grid_threads()) {
    const long long w = weight == 0 ? (long long)s.qd[i] : s.contig_off[i + 1] - s.contig_off[i];
    key[i] = kmax - (unsigned long long)w;
    val[i] = (int32_t)i;
  }
}

// Per tile and digit, the keys of the tile with that digit, stored digit-major
// (hist[d * tiles + t]) so that one exclusive scan gives every scatter base.
__global__ void k_sort_hist(const unsigned long long* key, long long C, int pass, unsigned* hist, long long tiles) {
  __shared__ unsigned cnt[256];
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    for (int d = threadIdx.x; d < 256; d += blockDim.x) cnt[d] = 0;
    __syncthreads();
    for (int k = 0; k < kSortItems; ++k) {
      const long long i = t * kSortTile + k * kBlock + threadIdx.x;
      if (i < C) atomicAdd(&cnt[digit_of(key[i], pass)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += blockDim.x) hist[(long long)d * tiles + t] = cnt[d];
    __syncthreads();
  }
}

struct HistLoad {
  const unsigned* h;
  __device__ unsigned long long operator()(long long i) const { return h[i]; }
};
struct HistStore {
  unsigned long long* base;
  __device__ void item(long long i, unsigned long long e) const { base[i] = e; }
  __device__ void last(long long, unsigned long long) const {}
};

// Stable scatter. A tile's keys are taken in index order, 256 per round; a
// key's place is its digit's base for the tile, plus the keys with that digit
// in earlier rounds, in earlier warps of this round and in earlier lanes.
__global__ void k_sort_scatter(const unsigned long long* key_in, const int32_t* val_in, unsigned long long* key_out,
                               int32_t* val_out, long long C, int pass, const unsigned long long* base,
                               long long tiles) {
  __shared__ unsigned running[256];
  __shared__ unsigned wcnt[kBlock / 32][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    for (int d = threadIdx.x; d < 256; d += blockDim.x) running[d] = 0;
    for (int k = 0; k < kSortItems; ++k) {
      const long long i = t * kSortTile + k * kBlock + threadIdx.x;
      const bool valid = i < C;
      const unsigned long long kk = valid ? key_in[i] : 0ull;
      const unsigned d = valid ? digit_of(kk, pass) : 256u + lane;   // no two invalid lanes match
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const unsigned before_lane = __popc(peers & ((1u << lane) - 1u));
      for (int x = threadIdx.x; x < (kBlock / 32) * 256; x += blockDim.x) (&wcnt[0][0])[x] = 0;
      __syncthreads();
      if (valid && before_lane == 0) wcnt[warp][d] = __popc(peers);
      __syncthreads();
      if (valid) {
        unsigned before_warp = 0;
        for (int w = 0; w < warp; ++w) before_warp += wcnt[w][d];
        const unsigned long long pos = base[(long long)d * tiles + t] + running[d] + before_warp + before_lane;
        key_out[pos] = kk;
        val_out[pos] = val_in[i];
      }
      __syncthreads();
      for (int dd = threadIdx.x; dd < 256; dd += blockDim.x) {
        unsigned sum = 0;
        for (int w = 0; w < kBlock / 32; ++w) sum += wcnt[w][dd];
        running[dd] += sum;
      }
      __syncthreads();
    }
  }
}

// One warp. A part is the key (weight sum << part_bits) | part index, so that
// the smallest key is the least-loaded part, the lowest index on ties, and no
// two keys are equal. Lane l holds the keys of parts l + 32 j, j < KPL, in
// registers. Per contig the warp takes the smallest key overall with the
// redux unit (one 32-bit minimum when every key fits in 32 bits, else the
// high halves, then the low halves at that high half) and the part holding
// it adds the contig's weight; no branch depends on the data.
template <int KPL, bool Narrow>
__global__ void __launch_bounds__(32) k_lpt_assign(const unsigned long long* key, const int32_t* val, long long C,
                                                   unsigned long long kmax, int P, int part_bits, int32_t* part,
                                                   int64_t* psum) {
  const unsigned full = 0xffffffffu;
  const unsigned long long idx_mask = (1ull << part_bits) - 1;
  const int lane = threadIdx.x;
  unsigned long long K[KPL];
#pragma unroll
  for (int j = 0; j < KPL; ++j) K[j] = lane + 32 * j < P ? (unsigned long long)(lane + 32 * j) : ~0ull;
  for (long long i0 = 0; i0 < C; i0 += 32) {
    const long long ii = i0 + lane;
    const int32_t ci = ii < C ? val[ii] : -1;
    const unsigned long long w = ii < C ? (kmax - key[ii]) << part_bits : 0ull;
    unsigned long long mine = 0;
    const int cnt = (int)min(32ll, C - i0);
    for (int q = 0; q < cnt; ++q) {
      const unsigned long long wq = __shfl_sync(full, w, q);
      unsigned long long my = K[0];
#pragma unroll
      for (int j = 1; j < KPL; ++j) my = min(my, K[j]);
      unsigned long long m;
      if (Narrow) {
        m = __reduce_min_sync(full, (unsigned)min(my, 0xffffffffull));
      } else {
        const unsigned hi = (unsigned)(my >> 32);
        const unsigned mhi = __reduce_min_sync(full, hi);
        const unsigned mlo = __reduce_min_sync(full, hi == mhi ? (unsigned)my : 0xffffffffu);
        m = ((unsigned long long)mhi << 32) | mlo;
      }
      mine = lane == q ? m : mine;
#pragma unroll
      for (int j = 0; j < KPL; ++j) K[j] += K[j] == m ? wq : 0ull;
    }
    if (ii < C) part[ci] = (int32_t)(mine & idx_mask);
  }
#pragma unroll
  for (int j = 0; j < KPL; ++j)
    if (lane + 32 * j < P) psum[lane + 32 * j] = (int64_t)(K[j] >> part_bits);
}

template <int KPL>
void lpt_launch(bool narrow, const unsigned long long* key, const int32_t* val, long long C, unsigned long long kmax,
                int P, int part_bits, int32_t* part, int64_t* psum, cudaStream_t st) {
  if (narrow) k_lpt_assign<KPL, true><<<1, 32, 0, st>>>(key, val, C, kmax, P, part_bits, part, psum);
  else k_lpt_assign<KPL, false><<<1, 32, 0, st>>>(key, val, C, kmax, P, part_bits, part, psum);
}

}  // namespace

cudaError_t launch_partition(const Scratch& s, long long C, int weight, long long max_weight, int P,
                             const SortBuffers& b, int32_t* part, int64_t* psum, const LaunchEnv& env) {
  int bits = 8;
  while (bits < 63 && (max_weight >> bits) != 0) bits += 8;
  const unsigned long long kmax = bits >= 64 ? ~0ull : (1ull << bits) - 1;
  if (C > 0) {
    const long long tiles = (C + kSortTile - 1) / kSortTile;
    const long long nh = 256 * tiles;
    const long long scan_tiles = (nh + kTileItems - 1) / kTileItems;
    if (scan_tiles > b.state_cap || tiles > b.tiles_cap) return cudaErrorInvalidValue;
    k_sort_keys<<<grid_for(C, env), kBlock, 0, env.stream>>>(s, C, weight, kmax, b.key[0], b.val[0]);
    mark(env, "k_sort_keys");
    const int grid = (int)std::min<long long>(tiles, (long long)env.num_sms * 4);
    int cur = 0;
    for (int pass = 0; pass < bits / 8; ++pass) {
      k_sort_hist<<<grid, kBlock, 0, env.stream>>>(b.key[cur], C, pass, b.hist, tiles);
      mark(env, "k_sort_hist");
      cudaMemsetAsync(b.state, 0, (size_t)(b.state_cap + 1) * sizeof(unsigned long long), env.stream);
      k_scan<<<scan_grid(scan_tiles, env), kBlock, 0, env.stream>>>(HistLoad{b.hist}, HistStore{b.base}, nh,
                                                              b.state, b.state_cap, s.derr, K_SORT);
      mark(env, "k_scan_digits");
      k_sort_scatter<<<grid, kBlock, 0, env.stream>>>(b.key[cur], b.val[cur], b.key[cur ^ 1], b.val[cur ^ 1], C,
                                                      pass, b.base, tiles);
      mark(env, "k_sort_scatter");
      cur ^= 1;
    }
    int part_bits = 0;
    while ((1 << part_bits) < P) ++part_bits;
    if (part_bits + bits > 63) return cudaErrorInvalidValue;
    // narrow: the largest key, max_weight << part_bits | (P - 1), stays below 2^32 - 1
    const bool narrow = (((unsigned long long)max_weight << part_bits) | (unsigned long long)(P - 1)) < 0xffffffffull;
    const unsigned long long* kk = b.key[cur];
    const int32_t* vv = b.val[cur];
    if (P <= 32) lpt_launch<1>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    else if (P <= 64) lpt_launch<2>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    else if (P <= 128) lpt_launch<4>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    else if (P <= 256) lpt_launch<8>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    else if (P <= 512) lpt_launch<16>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    else lpt_launch<32>(narrow, kk, vv, C, kmax, P, part_bits, part, psum, env.stream);
    mark(env, "k_lpt_assign");
  } else {
    cudaMemsetAsync(psum, 0, (size_t)P * sizeof(int64_t), env.stream);
  }
  return cudaGetLastError();
}

}  // namespace cg
