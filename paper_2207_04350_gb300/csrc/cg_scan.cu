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
#include "cg_stage.cuh"

namespace cg {

namespace {

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
// with_cycles: the closed chains come first, on the same (cooperative) grid, when
// there are any.
__global__ void __launch_bounds__(kBlock) k_heads(DevGraph g, Scratch s, bool with_cycles, int64_t* user_off,
                                                  long long user_cap) {
  pdl_enter();
  __shared__ unsigned long long tot[2][kBlock / 32];   // the prefix's sums, the words' sums
  const long long n = g.n;
  const bool stop = gave_up(s.derr);
  const unsigned cyc = with_cycles ? *(volatile unsigned*)&s.ctr->n_cycle_reads : 0u;   // the same for every block
  if (__syncthreads_or(stop)) return;
  if (cyc > 0) {
    Counters* c = s.ctr;
    auto sync = [&] { return grid_sync(c, s.derr, gridDim.x); };
    if (!close_cycles(g, s, cyc, grid_tid(), grid_threads(), sync) || !sync()) return;
  }
  for (long long i = grid_tid(); i <= s.scan_tiles_cap; i += grid_threads()) s.scan_state[i] = 0ull;   // of the piece scan
  const int tid = threadIdx.x;
  for (int tile = (int)blockIdx.x; tile < s.h_tiles; tile += (int)gridDim.x) {   // block-uniform
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
        run = block_sum<kBlock / 32>(run, tot[1]);
        first = false;
      }
      unsigned long long all;
      const unsigned long long e =
          run + block_exclusive<kBlock / 32>(((unsigned long long)__popc(bits) << kHeadShift) | reads, tot[0], &all);
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
    if (tile == s.h_tiles - 1 && tid == 0) {
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
}

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
  const bool stop = gave_up(s.derr);
  const long long W = *(const volatile unsigned*)&s.ctr->n_walk;
  if (__syncthreads_or(stop)) return;
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
    unsigned long long all, e = block_exclusive<kBlock / 32>(sum, tot, &all);
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

__global__ void k_scatter(DevGraph g, Scratch s) {
  pdl_enter();
  scatter_reads(g, s, gave_up(s.derr), grid_tid(), grid_threads());
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
  if (gave_up(s.derr)) return;
  if (C + 1 > cap) {
    if (grid_tid() == 0) set_error(s.derr, DERR_CAPACITY, K_CONTIG_OFF, C + 1);
    return;
  }
  for (long long i = grid_tid(); i <= C; i += grid_threads()) out[i] = s.contig_off[i];
}

}  // namespace

cudaError_t launch_offsets(const DevGraph& g, const Scratch& s, const Tuning& t, const LaunchEnv& env,
                           int64_t* user_off, long long user_cap, bool with_cycles) {
  if (g.n == 0) {
    k_contig_off<<<1, kBlock, 0, env.stream>>>(s);
    mark(env, "k_contig_off");
    return cudaGetLastError();
  }
  if (s.small) return launch_small(g, s, t, kStageOffsets, user_off, user_cap, env, env.pdl_first);
  cudaError_t e = cudaSuccess;
  if (with_cycles) {
    // as many blocks as the closed chains, of oriented candidates, or the tiles can use
    const long long need = std::max((2 * most_candidates(g) + kBlock - 1) / kBlock, (long long)s.h_tiles);
    static const int heads_resident = resident_blocks(k_heads);
    const long long most = std::min<long long>(env.coop_blocks, (long long)env.num_sms * heads_resident);
    DevGraph gg = g;
    Scratch sc = s;
    void* args[] = {&gg, &sc, &with_cycles, &user_off, &user_cap};
    e = coop((const void*)k_heads, (int)std::max(1LL, std::min(most, need)), args, env, env.pdl_first);
  } else {
    e = launch_k(k_heads, s.h_tiles, env, env.pdl_first, g, s, with_cycles, user_off, user_cap);
  }
  if (e != cudaSuccess) return e;
  mark(env, "k_heads");
  static const int scatter_resident = resident_blocks(k_scatter);   // a persistent grid
  const long long spelled = most_spelled(g), scatter_need = (spelled + kBlock * kScatterItems - 1) / (kBlock * kScatterItems);
  e = launch_k(k_scatter, (int)std::max(1LL, std::min((long long)env.num_sms * scatter_resident, scatter_need)), env,
               true, g, s);
  if (e != cudaSuccess) return e;
  mark(env, "k_scatter");
  PieceStore ps{s.out_off, s.contig_off, s.tile_seg, s.tiles_cap, t.tile_bytes, s.ctr, s.derr, user_off, user_cap};
  e = launch_k(k_pieces, (int)std::max(1LL, std::min((spelled + kPieceTile - 1) / kPieceTile, (long long)env.num_sms * 4)),
               env, true, s, ps);
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
// The sort is a stable LSD radix sort, 8-bit digits, of kmax - weight, in one
// block for up to 65,536 contigs; the assignment is sequential by definition
// and runs in one block, a round of up to one contig per part at a time.
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
                               long long tiles, const DevError* derr) {
  if (gave_up(derr)) return;                         // the scan did: base is not whole
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

// The same sort by one block, for at most kSortBlockMax contigs, where the
// launches and round trips of the kernels above are what a pass costs. Each of
// the 32 warps takes a run of the keys, counts its digits, and after one scan
// over digits and warps writes its keys in order, so the sort is stable; eight
// keys per lane are loaded before any is used. It sorts by wmax - weight, wmax
// the largest weight there is, so that small weights (reads per contig) need
// fewer passes than the bound kmax. Results in key[0], val[0]. The 3.1 Gb
// graph's 13,124 contigs by reads, one pass: 27 us by events (40 in two passes of
// eight bits), and 100 for the ten launches above; by bases, three passes, 66 and
// 136. The line (kSortBlockMax) lies between where the block's passes, which grow with
// the contigs, meet the launches by reads and by bases, block / launches: 32,000
// contigs 40 / 99 and, in two passes, 89 / 138; 49,000 56 / 101 and 128 / 138; 65,000
// 72 / 101 and 165 / 137; 98,000 102 / 102 and 240 / 139.
constexpr int kSortBlock = 1024;
constexpr int kSortLoad = 8;
constexpr int kSortBits = 10, kSortDigits = 1 << kSortBits;   // a digit per thread in the scan
constexpr int kSortSmem = kSortBlock / 32 * kSortDigits * 4;  // counts per warp and digit

__device__ __forceinline__ unsigned wide_digit(unsigned long long key, int pass) {
  return (unsigned)((key >> (kSortBits * pass)) & (unsigned long long)(kSortDigits - 1));
}

__global__ void __launch_bounds__(kSortBlock) k_sort_block(const Scratch s, int C, int weight, unsigned long long kmax,
                                                           unsigned long long* key0, unsigned long long* key1,
                                                           int32_t* val0, int32_t* val1) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char staged[];
  unsigned(*const cnt)[kSortDigits] = reinterpret_cast<unsigned(*)[kSortDigits]>(staged);
  __shared__ unsigned long long red[kSortBlock / 32];
  __shared__ unsigned warp_tot[kSortBlock / 32];
  const unsigned full = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  auto weight_of = [&](int i) -> unsigned long long {
    return weight == 0 ? (unsigned long long)s.qd[i] : (unsigned long long)(s.contig_off[i + 1] - s.contig_off[i]);
  };
  unsigned long long wmax = 0;
#pragma unroll 8
  for (int i = tid; i < C; i += kSortBlock) wmax = max(wmax, weight_of(i));
  for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(full, wmax, o));
  if (lane == 0) red[warp] = wmax;
  __syncthreads();
  wmax = red[lane];
  for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(full, wmax, o));
  int passes = 1;
  while (passes < 7 && (wmax >> (kSortBits * passes)) != 0) ++passes;
  const int seg = (C + kSortBlock - 1) / kSortBlock * 32;          // keys per warp, whole rounds of 32
  const int i_begin = warp * seg, i_end = min(C, i_begin + seg);
  for (int pass = 0; pass < passes; ++pass) {
    const bool to0 = ((passes - pass) & 1) != 0;                   // the last pass writes buffer 0
    const unsigned long long* kin = to0 ? key1 : key0;
    const int32_t* vin = to0 ? val1 : val0;
    unsigned long long* kout = to0 ? key0 : key1;
    int32_t* vout = to0 ? val0 : val1;
    // a key as sorted; the last pass stores kmax - weight
    auto load = [&](int i) -> unsigned long long { return pass == 0 ? wmax - weight_of(i) : kin[i]; };
    const unsigned long long shift = pass == passes - 1 ? kmax - wmax : 0ull;
    for (int w = 0; w < kSortBlock / 32; ++w) cnt[w][tid] = 0;
    __syncthreads();
    for (int i0 = i_begin; i0 < i_begin + seg; i0 += 32 * kSortLoad) {   // warp-uniform
      unsigned long long k[kSortLoad];
#pragma unroll
      for (int j = 0; j < kSortLoad; ++j) k[j] = i0 + 32 * j + lane < i_end ? load(i0 + 32 * j + lane) : 0ull;
#pragma unroll
      for (int j = 0; j < kSortLoad; ++j)
        if (i0 + 32 * j + lane < i_end) atomicAdd(&cnt[warp][wide_digit(k[j], pass)], 1u);
    }
    __syncthreads();
    {                                                              // exclusive sums by digit, then by warp
      unsigned sum = 0;
#pragma unroll 8
      for (int w = 0; w < kSortBlock / 32; ++w) sum += cnt[w][tid];
      unsigned inc = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += x;
      }
      if (lane == 31) warp_tot[warp] = inc;
      __syncthreads();
      unsigned run = inc - sum;
      for (int w = 0; w < warp; ++w) run += warp_tot[w];
#pragma unroll 8
      for (int w = 0; w < kSortBlock / 32; ++w) {
        const unsigned c = cnt[w][tid];
        cnt[w][tid] = run;
        run += c;
      }
    }
    __syncthreads();
    for (int i0 = i_begin; i0 < i_begin + seg; i0 += 32 * kSortLoad) {
      unsigned long long k[kSortLoad];
      int32_t v[kSortLoad];
#pragma unroll
      for (int j = 0; j < kSortLoad; ++j) {
        const int i = i0 + 32 * j + lane;
        k[j] = i < i_end ? load(i) : 0ull;
        v[j] = i < i_end ? (pass == 0 ? i : vin[i]) : 0;
      }
#pragma unroll
      for (int j = 0; j < kSortLoad; ++j) {
        const bool valid = i0 + 32 * j + lane < i_end;
        const unsigned d = wide_digit(k[j], pass);
        // the lanes with this digit: a ballot per bit (a match instruction per 32
        // keys and phase made the two passes 48 us)
        unsigned peers = __ballot_sync(full, valid);
#pragma unroll
        for (int b = 0; b < kSortBits; ++b) {
          const unsigned set = __ballot_sync(full, (d >> b) & 1u);
          peers &= (d >> b) & 1u ? set : ~set;
        }
        const unsigned at = valid ? cnt[warp][d] + __popc(peers & lt) : 0u;
        __syncwarp();
        if (valid && (peers & lt) == 0) cnt[warp][d] += __popc(peers);
        __syncwarp();
        if (valid) {
          kout[at] = k[j] + shift;
          vout[at] = v[j];
        }
      }
    }
    __syncthreads();
  }
}

// The assignment, a round of contigs at a time. A part is the key (weight sum
// << part_bits) | part index, so that the smallest key is the least-loaded
// part, the lowest index on ties, and no two keys are equal. Taken one by one,
// the next contigs go to the parts of rank 0, 1, 2, ... for as long as no part
// that has just received one is below the next rank's key: mostly for a whole
// round of P contigs, since the weights come in descending order and a round
// levels the sums. So a round ranks the P keys, hands contig r to the part of
// rank r and keeps the longest prefix for which that holds: all of it when every
// raised key is above the largest old one, else up to the first rank whose old
// key is above a raised key of a lower rank. When that is few (lpt_few), or not all for
// some rounds on end, a few parts lie below the others (which hold contigs larger than
// a share, say) and take the next contigs among themselves for long: one warp then
// hands kLptLeast contigs, and twice as many each further time in a row, to the
// smallest of the kLptLow lowest keys one by one, while that is below the next key.
// The parts are those of the rule taken literally.
// G threads per part, each comparing its key with a G-th of the P keys in shared
// memory. What bounds it is the chain of ranks and barriers of each round. A few
// parts, whose rounds would hand out that few contigs, take another way below.
// The 3.1 Gb graph's contigs into 72 / 128 / 1024 parts: 118 / 90 / 300 us by
// events, and 770 / 770 / 4851 one contig at a time in one warp. 20,000 contigs of a
// few reads behind so many large ones that 2 / 10 / 18 / 24 parts of 72 / 72 / 128 /
// 1024 lie below the others, whole call: 0.56 / 0.78 / 0.94 / 3.2 ms, 0.97 / 1.24 /
// 1.44 / 13.2 in rounds of as few and 1.31 / 1.31 / 1.31 / 8.0 one at a time.
constexpr int kLptLow = 64, kLptLeast = 48, kLptRun = 1024;
// Below this a round costs more than as many contigs one by one (27 to 40 ns each): a
// round is 0.65 us with up to 64 parts, 1.3 with 128, 16 with 1024.
__device__ __forceinline__ int lpt_few(int P) { return P > 256 ? kLptLow : P > 128 ? 32 : min(24, 3 * P / 4); }
constexpr int kLptSmem = 160 << 10;  // bytes of weights and parts staged at a time; kMaxParts contigs at least

// The smallest value of the lanes before this one.
template <typename K>
__device__ __forceinline__ K warp_min_before(K m, int lane) {
  const K none = ~(K)0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const K x = __shfl_up_sync(0xffffffffu, m, o);
    if (lane >= o) m = min(m, x);
  }
  const K e = __shfl_up_sync(0xffffffffu, m, 1);
  return lane == 0 ? none : e;
}

// The smallest value of a warp's lanes, by the redux unit.
__device__ __forceinline__ uint32_t warp_smallest(uint32_t x) { return __reduce_min_sync(0xffffffffu, x); }
__device__ __forceinline__ unsigned long long warp_smallest(unsigned long long x) {
  const unsigned hi = (unsigned)(x >> 32), mhi = __reduce_min_sync(0xffffffffu, hi);
  return ((unsigned long long)mhi << 32) | __reduce_min_sync(0xffffffffu, hi == mhi ? (unsigned)x : ~0u);
}

// Contigs of weights w[0..most) one after another to the smallest of a warp's keys, k0
// and (kTwo) k1 of each lane, while that is below `limit`: the parts they go to in `to`,
// how many they are returned. 32 at a time have their weights and parts in registers.
template <bool kTwo, typename K>
__device__ __forceinline__ int lpt_one_by_one(const K* w, short* to, int most, K& k0, K& k1, K limit, int part_bits,
                                              int lane) {
  const unsigned mask = (1u << part_bits) - 1u;
  int q = 0;
  for (bool low = true; low && q < most;) {
    const int len = min(32, most - q);
    const K wl = lane < len ? w[q + lane] : (K)0;
    unsigned got = 0;
    int i = 0;
#pragma unroll 4
    for (; i < len; ++i) {
      const K wi = __shfl_sync(0xffffffffu, wl, i), m = warp_smallest(kTwo ? min(k0, k1) : k0);
      low = m < limit;
      if (!low) break;
      got = lane == i ? (unsigned)m & mask : got;
      k0 += k0 == m ? wi : (K)0;
      if (kTwo) k1 += k1 == m ? wi : (K)0;
    }
    if (lane < i) to[q + lane] = (short)got;
    q += i;
  }
  return q;
}

// How many of a g-th of the n4 keys are below `mine`.
template <int kUnroll>
__device__ __forceinline__ int keys_below(const uint32_t* keys, int n4, int g, int G, uint32_t mine) {
  int r0 = 0, r1 = 0;
#pragma unroll kUnroll
  for (int j = 4 * g; j < n4; j += 4 * G) {
    const uint4 x = *reinterpret_cast<const uint4*>(keys + j);
    r0 += (x.x < mine) + (x.y < mine);
    r1 += (x.z < mine) + (x.w < mine);
  }
  return r0 + r1;
}
template <int kUnroll>
__device__ __forceinline__ int keys_below(const unsigned long long* keys, int n4, int g, int G, unsigned long long mine) {
  int r0 = 0, r1 = 0;
#pragma unroll kUnroll
  for (int j = 2 * g; j < n4; j += 2 * G) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(keys + j);
    r0 += x.x < mine;
    r1 += x.y < mine;
  }
  return r0 + r1;
}

// A barrier of the first `count` threads of the block, whole warps, and the same
// with the or of a predicate over them.
__device__ __forceinline__ void part_sync(int count) { asm volatile("barrier.cta.sync 1, %0;" ::"r"(count) : "memory"); }
__device__ __forceinline__ bool part_sync_or(int count, bool x) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %2, 0;\n\tbarrier.cta.red.or.pred q, 1, %1, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(count), "r"((int)x)
      : "memory");
  return r != 0;
}

// G threads per part (a power of two): the first P * G threads, in whole warps,
// assign, and the others only stage weights and write parts. kUnroll: of the comparing
// loop, which is a handful of steps with few parts (72 parts by reads: 171 us a call
// with 1, 182 with 4; 1,024 parts 370 and 355).
template <typename K, int kUnroll>
__global__ void __launch_bounds__(kMaxParts, 1) k_lpt_assign(const unsigned long long* key, const int32_t* val, long long C,
                                                          unsigned long long kmax, int P, int G, int part_bits,
                                                          int chunk, int32_t* part, int64_t* psum,
                                                          const DevError* derr) {
  pdl_enter();
  if (gave_up(derr)) return;                               // a scan of the sort did: val is not whole
  __shared__ __align__(16) K keys[kMaxParts];              // by part
  __shared__ K old_key[kMaxParts], new_key[kMaxParts];     // by rank
  extern __shared__ __align__(16) unsigned char staged[];
  K* const w = reinterpret_cast<K*>(staged);               // chunk weights
  short* const to = reinterpret_cast<short*>(w + chunk);   // and the parts they go to
  __shared__ K warp_min[32], top;
  __shared__ int first_bad, handed, stop;
  __shared__ int again, run, bad_end;                      // rounds that kept a part on end, the next run, where the last one ended
  const unsigned full = 0xffffffffu;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const K none = ~(K)0;
  const int me = tid / G, g = tid & (G - 1);
  const bool act = me < P, lead = act && g == 0;
  const int n4 = (P + 3) & ~3, A = (P * G + 31) & ~31;
  if (tid >= P && tid < n4) keys[tid] = none;              // the last vector's empty places
  if (tid == 0) {
    again = 0;
    run = kLptLeast;
    bad_end = -1;
  }
  K mine = act ? (K)me : none;
  for (long long c0 = 0; c0 < C;) {
    const int n = (int)min((long long)chunk, C - c0);
#pragma unroll 8
    for (int i = tid; i < n; i += T) w[i] = (K)((kmax - key[c0 + i]) << part_bits);
    __syncthreads();
    const bool last = c0 + n == C;
    int cur = 0;
    if (tid < A) {
      while (cur < n && (last || n - cur >= P)) {            // the same for every thread of the parts
        const int cnt = min(P, n - cur);
        if (lead) keys[me] = mine;
        part_sync(A);
        int r = act ? keys_below<kUnroll>(keys, n4, g, G, mine) : 0;
        for (int o = G >> 1; o > 0; o >>= 1) r += __shfl_xor_sync(full, r, o);
        if (!act) r = P;
        const K raised = r < cnt ? mine + w[cur + r] : none;
        if (lead && r == cnt - 1) top = mine;
        part_sync(A);
        if (!part_sync_or(A, r < cnt - 1 && raised < top)) {
          if (r < cnt) {
            if (lead) to[cur + r] = (short)me;
            mine = raised;
          }
          cur += cnt;
          continue;
        }
        if (lead) {
          old_key[r] = mine;
          if (r < cnt) new_key[r] = raised;
        }
        if (tid == 0) {
          first_bad = cnt;
          again = cur == bad_end ? again + 1 : 0;
        }
        part_sync(A);
        const K m = tid < cnt ? new_key[tid] : none;         // thread t now looks at rank t
        K before = warp_min_before(m, lane);
        if (lane == 31) warp_min[warp] = min(before, m);
        part_sync(A);
        for (int x = 0; x < warp; ++x) before = min(before, warp_min[x]);
        if (tid > 0 && tid < cnt && old_key[tid] > before) atomicMin(&first_bad, tid);
        part_sync(A);
        const int kept = first_bad;
        if (kept >= (again < 3 ? lpt_few(P) : max(lpt_few(P), min(24, P)))) {   // again: no full round for a while
          if (r < kept) {
            if (lead) to[cur + r] = (short)me;
            mine = raised;
          }
          cur += kept;
          if (tid == 0) {
            run = kLptLeast;
            bad_end = cur;
          }
          continue;
        }
        if (warp == 0) {                                     // lane l: the parts of rank l and l + 32
          K k0 = lane < P ? old_key[lane] : none, k1 = lane + 32 < P ? old_key[lane + 32] : none;
          const K limit = P > kLptLow ? old_key[kLptLow] : none;
          const int most = min(__shfl_sync(full, run, 0), n - cur);
          const int q = P <= 32 ? lpt_one_by_one<false>(w + cur, to + cur, most, k0, k1, limit, part_bits, lane)
                                : lpt_one_by_one<true>(w + cur, to + cur, most, k0, k1, limit, part_bits, lane);
          new_key[lane] = k0;
          new_key[lane + 32] = k1;
          if (lane == 0) {
            handed = q;
            run = min(2 * run, kLptRun);
            bad_end = cur + q;
          }
        }
        part_sync(A);
        if (act && r < kLptLow) mine = new_key[r];
        cur += handed;
      }
      if (tid == 0) stop = cur;
    }
    __syncthreads();
    cur = stop;
#pragma unroll 8
    for (int i = tid; i < cur; i += T) part[val[c0 + i]] = to[i];
    c0 += cur;
    __syncthreads();
  }
  if (lead) psum[me] = (int64_t)(mine >> part_bits);
}

// Few parts, one contig after another, by one warp; the block's other warps only
// stage weights and write parts. Up to 4 parts (M > 0) the keys are kept sorted in
// registers, M of them: each contig goes to the first, whose raised key x moves to
// its place among the others, R[j] = min(R[j+1], max(R[j], x)), all places at once,
// so from one contig to the next it is an addition, a maximum and a minimum. Every
// lane does the same, which spares the warp any exchange. With more parts a lane
// holds one and the warp takes the smallest key with the redux unit. Either keeps
// its keys relative to the smallest sum, which it lifts out after every few
// contigs: no sum ever is further above the smallest than the largest weight, so
// they fit 32 bits unless that weight (w0) is huge, and the warp then takes 64-bit
// keys. Contigs of the 3.1 Gb graph by reads, 2 / 4 / 8 / 16 / 24 parts, by events:
// sorted 232 / 265 / 397 us, a part per lane 330 for any number, in rounds 1612 /
// 860 / 439 / 322 / 254 (by bases 385 at 16 and 358 at 20 parts, hence the line).
constexpr int kLptSorted = 4, kLptWarp = 19;

template <int M>
__global__ void __launch_bounds__(kBlock) k_lpt_few(const unsigned long long* key, const int32_t* val, long long C,
                                                    unsigned long long kmax, int P, int part_bits, int chunk,
                                                    int32_t* part, int64_t* psum, const DevError* derr) {
  pdl_enter();
  if (gave_up(derr)) return;                           // a scan of the sort did: val is not whole
  extern __shared__ __align__(16) unsigned char staged[];
  unsigned long long* const w = reinterpret_cast<unsigned long long*>(staged);
  short* const to = reinterpret_cast<short*>(w + chunk);
  const unsigned full = 0xffffffffu, none = ~0u;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned mask = (1u << part_bits) - 1u;
  constexpr int kAhead = M ? 8 : 32;                   // contigs between two lifts
  const unsigned long long w0 = kmax - key[0];         // the largest weight
  const bool narrow = w0 < (1ull << 32) && ((kAhead + 1) * w0 + 1) << part_bits < (1ull << 32);
  unsigned R[M ? M : 1];                               // sorted keys, or this lane's
#pragma unroll
  for (int j = 0; j < M; ++j) R[j] = j < P ? (unsigned)j : none;
  if (M == 0) R[0] = lane < P ? (unsigned)lane : none;
  unsigned long long lifted = 0;                       // taken out of every sum so far
  unsigned long long wide = lane < P ? (unsigned long long)lane : ~0ull;   // this lane's key when 32 bits do not hold them
  for (long long c0 = 0; c0 < C; c0 += chunk) {
    const int n = (int)min((long long)chunk, C - c0);
#pragma unroll 8
    for (int i = tid; i < n; i += kBlock) w[i] = kmax - key[c0 + i];
    __syncthreads();
    if (tid < 32 && !narrow) {
      for (int i0 = 0; i0 < n; i0 += 32) {
        const unsigned long long wl = i0 + lane < n ? w[i0 + lane] << part_bits : 0ull;
        unsigned got = 0;
        for (int q = 0; q < min(32, n - i0); ++q) {
          const unsigned long long wq = __shfl_sync(full, wl, q);
          const unsigned hi = (unsigned)(wide >> 32), mhi = __reduce_min_sync(full, hi);
          const unsigned mlo = __reduce_min_sync(full, hi == mhi ? (unsigned)wide : none);
          const unsigned long long m = ((unsigned long long)mhi << 32) | mlo;
          got = lane == q ? mlo & mask : got;
          wide += wide == m ? wq : 0ull;
        }
        if (i0 + lane < n) to[i0 + lane] = (short)got;
      }
    } else if (tid < 32 && M == 0) {
      for (int i0 = 0; i0 < n; i0 += kAhead) {
        const unsigned wl = i0 + lane < n ? (unsigned)w[i0 + lane] << part_bits : 0u;
        unsigned got = 0, m = 0;
        for (int q = 0; q < min(32, n - i0); ++q) {
          const unsigned wq = __shfl_sync(full, wl, q);
          m = __reduce_min_sync(full, R[0]);
          got = lane == q ? m & mask : got;
          R[0] += R[0] == m ? wq : 0u;
        }
        if (i0 + lane < n) to[i0 + lane] = (short)got;
        const unsigned lift = __reduce_min_sync(full, R[0]) & ~mask;
        if (lane < P) R[0] -= lift;
        lifted += lift >> part_bits;
      }
    } else if (tid < 32) {
      for (int i0 = 0; i0 < n; i0 += kAhead) {
        unsigned wi[kAhead], got[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) wi[k] = i0 + k < n ? (unsigned)w[i0 + k] << part_bits : 0u;
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {             // past n a weight of 0 changes nothing
          got[k] = R[0] & mask;
          const unsigned x = R[0] + wi[k];
#pragma unroll
          for (int j = 0; j < M; ++j) {
            const unsigned above = j + 1 < M ? R[j + 1 < M ? j + 1 : j] : none;
            R[j] = min(above, j == 0 ? x : max(R[j], x));
          }
        }
        if (lane == 0)
#pragma unroll
          for (int k = 0; k < kAhead; ++k)
            if (i0 + k < n) to[i0 + k] = (short)got[k];
        const unsigned lift = R[0] & ~mask;
#pragma unroll
        for (int j = 0; j < M; ++j) R[j] -= j < P ? lift : 0u;
        lifted += lift >> part_bits;
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int i = tid; i < n; i += kBlock) part[val[c0 + i]] = to[i];
    __syncthreads();
  }
  if (tid >= 32) return;
  if (!narrow) {
    if (lane < P) psum[lane] = (int64_t)(wide >> part_bits);
  } else if (M == 0) {
    if (lane < P) psum[lane] = (int64_t)(lifted + (R[0] >> part_bits));
  } else if (lane == 0) {
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < P) psum[R[j] & mask] = (int64_t)(lifted + (R[j] >> part_bits));
  }
}

// One block with the contigs' weights and parts staged: as many at a time as fit
// kLptSmem, which is all of them for most graphs, since each chunk costs two round
// trips to memory.
int lpt_chunk(long long C, int weight_bytes) {
  const int most = kLptSmem / (weight_bytes + (int)sizeof(short)) / 64 * 64;
  return std::max(C < most ? (int)((C + 63) / 64 * 64) : most, kMaxParts);
}

template <typename... A, typename... B>
cudaError_t lpt_launch(void (*kernel)(A...), int chunk, int weight_bytes, int threads, const LaunchEnv& env, B... args) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLptSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)chunk * (size_t)(weight_bytes + (int)sizeof(short));
  cfg.stream = env.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = env.pdl && !(env.marks && env.marks->on) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One part takes every contig.
__global__ void __launch_bounds__(kBlock) k_lpt_one(const Scratch s, long long C, int weight, int32_t* part,
                                                    int64_t* psum) {
  unsigned long long sum = 0;
  for (long long i = grid_tid(); i < C; i += grid_threads()) {
    part[i] = 0;
    sum += weight == 0 ? (unsigned long long)s.qd[i] : (unsigned long long)(s.contig_off[i + 1] - s.contig_off[i]);
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(reinterpret_cast<unsigned long long*>(psum), sum);
}

}  // namespace

cudaError_t launch_partition(const Scratch& s, long long C, int weight, long long max_weight, int P,
                             const SortBuffers& b, int32_t* part, int64_t* psum, const LaunchEnv& env) {
  int bits = 8;
  while (bits < 63 && (max_weight >> bits) != 0) bits += 8;
  const unsigned long long kmax = bits >= 64 ? ~0ull : (1ull << bits) - 1;
  if (C <= 0 || P == 1) cudaMemsetAsync(psum, 0, (size_t)P * sizeof(int64_t), env.stream);
  if (C <= 0) return cudaGetLastError();
  if (P == 1) {
    k_lpt_one<<<grid_for(C, env), kBlock, 0, env.stream>>>(s, C, weight, part, psum);
    mark(env, "k_lpt_one");
    return cudaGetLastError();
  }
  int cur = 0;
  const bool small = C <= kSortBlockMax;
  if (small) {
    cudaError_t e = cudaFuncSetAttribute(k_sort_block, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortSmem);
    if (e != cudaSuccess) return e;
    k_sort_block<<<1, kSortBlock, kSortSmem, env.stream>>>(s, (int)C, weight, kmax, b.key[0], b.key[1], b.val[0],
                                                           b.val[1]);
    mark(env, "k_sort_block");
  } else {
    const long long tiles = (C + kSortTile - 1) / kSortTile;
    const long long nh = 256 * tiles;
    const long long scan_tiles = (nh + kTileItems - 1) / kTileItems;
    if (scan_tiles > b.state_cap || tiles > b.tiles_cap) return cudaErrorInvalidValue;
    k_sort_keys<<<grid_for(C, env), kBlock, 0, env.stream>>>(s, C, weight, kmax, b.key[0], b.val[0]);
    mark(env, "k_sort_keys");
    const int grid = (int)std::min<long long>(tiles, (long long)env.num_sms * 4);
    for (int pass = 0; pass < bits / 8; ++pass) {
      k_sort_hist<<<grid, kBlock, 0, env.stream>>>(b.key[cur], C, pass, b.hist, tiles);
      mark(env, "k_sort_hist");
      cudaMemsetAsync(b.state, 0, (size_t)(b.state_cap + 1) * sizeof(unsigned long long), env.stream);
      k_scan<<<scan_grid(scan_tiles, env), kBlock, 0, env.stream>>>(HistLoad{b.hist}, HistStore{b.base}, nh,
                                                              b.state, b.state_cap, s.derr, K_SORT);
      mark(env, "k_scan_digits");
      k_sort_scatter<<<grid, kBlock, 0, env.stream>>>(b.key[cur], b.val[cur], b.key[cur ^ 1], b.val[cur ^ 1], C,
                                                      pass, b.base, tiles, s.derr);
      mark(env, "k_sort_scatter");
      cur ^= 1;
    }
  }
  int part_bits = 0;
  while ((1 << part_bits) < P) ++part_bits;
  if (part_bits + bits > 63) return cudaErrorInvalidValue;
  // narrow: the largest key, max_weight << part_bits | (P - 1), stays below 2^32 - 1
  const bool narrow = (((unsigned long long)max_weight << part_bits) | (unsigned long long)(P - 1)) < 0xffffffffull;
  const unsigned long long* const kk = b.key[cur];
  const int32_t* const vv = b.val[cur];
  cudaError_t e;
  if (P <= kLptWarp) {
    auto* const kernel = P <= 2 ? k_lpt_few<2> : P <= kLptSorted ? k_lpt_few<4> : k_lpt_few<0>;
    const int chunk = lpt_chunk(C, 8);
    e = lpt_launch(kernel, chunk, 8, kBlock, env, kk, vv, C, kmax, P, part_bits, chunk, part, psum, s.derr);
  } else {
    // threads per part: as many as 512 threads allow, and no more than there are
    // vectors of keys (72 parts: 161 us with one, 125 with four, 131 with eight)
    int G = 1;
    while (2 * G * P <= 512 && 2 * G <= (P + 3) / 4) G *= 2;
    const int threads = std::max(256, (P * G + 31) & ~31);   // enough of them to stage the weights
    const int chunk = lpt_chunk(C, narrow ? 4 : 8);
    auto* const narrow_kernel = P <= 256 ? k_lpt_assign<uint32_t, 1> : k_lpt_assign<uint32_t, 4>;
    e = narrow ? lpt_launch(narrow_kernel, chunk, 4, threads, env, kk, vv, C, kmax, P, G, part_bits, chunk, part, psum,
                            s.derr)
               : lpt_launch(k_lpt_assign<unsigned long long, 4>, chunk, 8, threads, env, kk, vv, C, kmax, P, G, part_bits, chunk,
                            part, psum, s.derr);
  }
  if (e != cudaSuccess) return e;
  mark(env, "k_lpt_assign");
  return cudaGetLastError();
}

}  // namespace cg
