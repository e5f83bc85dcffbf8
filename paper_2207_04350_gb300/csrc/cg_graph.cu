// cg_graph.cu - graph stage of contig generation on sm_103a:
//   input checks, BranchRemoval (Alg. 2, Sec. 4.2), the oriented successor
//   table of the unbranched matrix L, and chain discovery by list ranking
//   (the GPU counterpart of ConnectedComponent + the walk order of
//   LocalAssembly, Sec. 4.2 and 4.4).
//
// Chains as linked lists. Every unmasked read v becomes two oriented reads
// x = 2v + o (o = 0 forward, 1 reverse complement). Oriented read (v,o) leaves
// v through end 1-o; if L has the overlap (v->w) on that end, its successor
// is (w, E_w), the orientation in which w is entered. Each chain thus appears
// as two directed lists, one the reverse of the other, and a closed chain as
// two directed cycles. (v,o) has a predecessor exactly when (v,1-o) has a
// successor.
//
// List ranking (Helman-JaJa style sublists): every list head and every read
// whose hash falls in a 2^-k sample starts a sublist; one thread walks each
// sublist to the next sublist start. Each list head then walks its (short)
// list of sublists twice -- once for the length, the tail and the smallest
// read, once to hand every sublist its distance to the tail. Lists with more
// sublists than that walk follows are left to grid-synchronised pointer
// jumping, which only runs when needed; closed chains (no head) go to their
// own kernel. A read then knows, from its two oriented copies, the chain's
// length, both end reads, its position from either end, and the chain's
// smallest read id.
//
// The mask stage lists the candidates (unmasked reads with overlaps, in
// candidate order c, with cidx[v] = c) and the chain stage indexes its records
// by candidate, oriented copies u = 2c + o: they sit together instead of
// spreading over arrays of n reads. Sublist records keep read ids, which the
// canonical order compares.
#include <cuda_runtime.h>

#include "cg_internal.cuh"
#include "cg_stage.cuh"

namespace cg {

namespace {

constexpr int kListWalkMax = 64;              // sublists a list head follows before leaving it to jumping
constexpr int kUnresolved = -2;               // pj next field of a sublist no list walk has finished

__device__ __forceinline__ int sampled(int v, int ruler_log2) {
  unsigned h = (unsigned)v * 0x9E3779B1u;
  h ^= h >> 15;
  h *= 0x85EBCA77u;
  h ^= h >> 13;
  return (h & ((1u << ruler_log2) - 1u)) == 0u;
}

// -------------------------------------------------------------- validation
__global__ void k_validate_reads(DevGraph g, DevError* c) {
  for (long long v = grid_tid(); v < g.n; v += grid_threads()) {
    int64_t a = rowp(g, v), b = rowp(g, v + 1);
    if (b < a) set_error(c, DERR_GRAPH, K_VALIDATE1, v);
    int32_t L = g.len[v];
    int64_t o = g.off[v];
    if (L < 1 || o < 0 || o + L > g.packed_bytes * 4) set_error(c, DERR_GRAPH, K_VALIDATE1, v);
  }
  if (grid_tid() == 0) {
    if (rowp(g, 0) != 0 || rowp(g, g.n) != g.m) set_error(c, DERR_GRAPH, K_VALIDATE1, -1);
  }
}

__global__ void k_validate_entries(DevGraph g, DevError* c) {
  // Row bounds are clamped to [0, m] so that a malformed row_ptr (reported by
  // k_validate_reads, which runs just before without a wait) reads nothing
  // outside the arrays.
  for (long long u = grid_tid(); u < g.n; u += grid_threads()) {
    int64_t a = max((int64_t)0, min(rowp(g, u), g.m)), b = max(a, min(rowp(g, u + 1), g.m));
    for (int64_t x = a; x < b; ++x) {
      int32_t v = g.col[x];
      uint8_t cd = g.code[x];
      if (v < 0 || v >= g.n || v == u || cd > 3) { set_error(c, DERR_GRAPH, K_VALIDATE2, x); continue; }
      if (g.pre) {                         // x-drop form: indices into the stored reads u and v
        const int32_t p = g.pre[x], q = g.post[x];
        if (p < 0 || p > g.len[u] - 1 || q < 0 || q > g.len[v] - 1) set_error(c, DERR_GRAPH, K_VALIDATE2, x);
      } else {
        const int32_t s = g.suf[x];
        if (s < 1 || s > g.len[v] - 1) set_error(c, DERR_GRAPH, K_VALIDATE2, x);
      }
      for (int64_t y = a; y < x; ++y)
        if (g.col[y] == v) set_error(c, DERR_GRAPH, K_VALIDATE2, x);
      int64_t va = max((int64_t)0, min(rowp(g, v), g.m)), vb = max(va, min(rowp(g, v + 1), g.m));
      int found = 0;
      uint8_t want = (uint8_t)(((cd & 1) << 1) | (cd >> 1));
      for (int64_t y = va; y < vb; ++y) {
        if (g.col[y] != u) continue;
        ++found;
        if (g.code[y] != want) set_error(c, DERR_GRAPH, K_VALIDATE2, x);
      }
      if (found != 1) set_error(c, DERR_GRAPH, K_VALIDATE2, x);
    }
  }
}

// ----------------------------------------------------------- BranchRemoval
// d[v] = row length of S (Sec. 4.2); d >= 3 is a branch. A read of degree
// <= 2 whose overlaps to reads of degree <= 2 are exactly two, both on the
// same end, cannot be passed by a valid walk and is a branch too. Reads with
// no overlap are lone reads: a one-read contig when min_chain <= 1. Every
// word of the mask-stage bitmap of contig heads is written here (the lone
// reads' bits); the chain stage adds the other heads to a copy of it.
// A warp owns 256 consecutive reads per pass, eight per lane: a lane loads
// its eight row starts with 16-byte loads (a read's degree is the next start
// minus its own; the eighth read's end is the next lane's first start),
// writes its eight branch bytes as one 8-byte store, and queues the reads of
// degree 1 or 2, whose rule needs the neighbours' degrees. The whole warp
// then resolves the queue together, so that a pass waits for three dependent
// loads (row starts; col and code; the neighbours' rows) whatever the mix of
// degrees in it. The candidate and lone-read lists gather in per-warp
// shared-memory buffers and reach the global lists with one reservation per
// block at the end (a warp flushes early only when a pass would overflow its
// buffer): returning atomics on one counter, one per pass, would serialise.
#ifndef CG_MASK_MIN_BLOCKS
#define CG_MASK_MIN_BLOCKS 4                   // resident blocks per SM the registers must allow
#endif
constexpr int kMaskLane = 8;                  // reads per lane per pass
constexpr int kMaskSpan = 32 * kMaskLane;     // reads per warp per pass
constexpr int kMaskWarps = kBlock / 32;
constexpr int kMaskBuf = 256;                 // buffered list entries per warp

template <typename RP>
__device__ __forceinline__ void load_rows(const RP* p, int64_t r[kMaskLane]);
template <>
__device__ __forceinline__ void load_rows<int64_t>(const int64_t* p, int64_t r[kMaskLane]) {
#pragma unroll
  for (int k = 0; k < kMaskLane / 2; ++k) {
    const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(p) + k);
    r[2 * k] = x.x;
    r[2 * k + 1] = x.y;
  }
}
template <>
__device__ __forceinline__ void load_rows<int32_t>(const int32_t* p, int64_t r[kMaskLane]) {
#pragma unroll
  for (int k = 0; k < kMaskLane / 4; ++k) {
    const int4 x = __ldg(reinterpret_cast<const int4*>(p) + k);
    r[4 * k] = x.x; r[4 * k + 1] = x.y; r[4 * k + 2] = x.z; r[4 * k + 3] = x.w;
  }
}

// Exclusive prefix of per-lane counts across the warp; the total in *tot.
__device__ __forceinline__ unsigned warp_exclusive(unsigned x, unsigned* tot, int lane) {
  unsigned inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  *tot = __shfl_sync(0xffffffffu, inc, 31);
  return inc - x;
}

// Appends n buffered entries of one warp to a global list with one atomic.
__device__ __forceinline__ void warp_flush(unsigned* counter, int32_t* list, const int32_t* buf, unsigned n,
                                           int lane) {
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(counter, n);
  base = __shfl_sync(0xffffffffu, base, 0);
  for (unsigned i = lane; i < n; i += 32) list[base + i] = buf[i];
}

// Reserves n entries of a global list for one warp (one atomic); returns the first.
__device__ __forceinline__ unsigned warp_reserve(unsigned* counter, unsigned n, int lane) {
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(counter, n);
  return __shfl_sync(0xffffffffu, base, 0);
}

// Candidates get their index when written out: cand[c] = v and cidx[v] = c.
__device__ __forceinline__ void flush_cands(const Scratch& s, const int32_t* buf, unsigned n, unsigned base,
                                            int lane) {
  for (unsigned i = lane; i < n; i += 32) {
    const int32_t v = buf[i];
    s.cand[base + i] = v;
    s.cidx[v] = (int32_t)(base + i);
  }
}

template <typename RP, bool kAligned>
__global__ void __launch_bounds__(kBlock, CG_MASK_MIN_BLOCKS) k_mask(DevGraph g, Scratch s) {
  pdl_enter();
  __shared__ int64_t q_row[kMaskWarps][kMaskSpan];   // queued reads: row start
  __shared__ uint16_t q_pos[kMaskWarps][kMaskSpan];  //   and position in the pass | (degree == 2) << 8
  __shared__ int32_t b_cand[kMaskWarps][kMaskBuf];   // buffered list entries
  __shared__ int32_t b_lone[kMaskWarps][kMaskBuf];
  __shared__ unsigned blk_n[2], blk_base[2];
  const RP* const rp = reinterpret_cast<const RP*>(g.row_ptr);
  Counters* c = s.ctr;
  if (threadIdx.x < 2) blk_n[threadIdx.x] = 0;       // read after the first barrier below
  unsigned long long nb = 0;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t* const bc = b_cand[wib];
  int32_t* const bl = b_lone[wib];
  unsigned nc = 0, nl = 0;                           // buffered entries (warp-uniform)
  const long long stride = (long long)gridDim.x * kMaskWarps * kMaskSpan;
  // The row starts of a pass (and, on lane 31, the start after its last read).
  // They are loaded one pass ahead, so that the next pass's stream of row_ptr
  // is in flight while this pass resolves its queued reads.
  const int p0 = kMaskLane * lane;
  auto load_pass = [&](long long wb, int64_t (&r)[kMaskLane], int64_t& e31) {
    const int cnt = (int)min((long long)kMaskSpan, g.n - wb);
    const bool full = cnt == kMaskSpan;
    if (kAligned && full) {
      load_rows<RP>(rp + wb + p0, r);
    } else {
#pragma unroll
      for (int j = 0; j < kMaskLane; ++j) r[j] = p0 + j <= cnt ? (int64_t)rp[wb + p0 + j] : 0;
    }
    e31 = lane == 31 && full ? (int64_t)rp[wb + kMaskSpan] : 0;
  };
  long long wbase = ((long long)blockIdx.x * kMaskWarps + wib) * kMaskSpan;
  int64_t r[kMaskLane], e31 = 0;
  if (wbase < g.n) load_pass(wbase, r, e31);
  for (; wbase < g.n; wbase += stride) {
    // warp-uniform trip count; row_ptr holds n + 1 entries
    const int cnt = (int)min((long long)kMaskSpan, g.n - wbase);
    const bool full = cnt == kMaskSpan;
    int64_t e = __shfl_down_sync(0xffffffffu, r[0], 1);
    if (lane == 31) e = e31;
    uint32_t br[2] = {0u, 0u};
    unsigned pend = 0, two = 0, lone = 0;
#pragma unroll
    for (int j = 0; j < kMaskLane; ++j) {
      const int64_t d = (j < kMaskLane - 1 ? r[j + 1] : e) - r[j];
      if (p0 + j < cnt) {
        if (d >= 3) { br[j >> 2] |= 1u << (8 * (j & 3)); ++nb; }
        else if (d > 0) { pend |= 1u << j; two |= (d == 2 ? 1u : 0u) << j; }
        else lone |= 1u << j;
      }
    }
    if (g.min_chain > 1) lone = 0;
    int64_t rn[kMaskLane], en31 = 0;                   // the next pass's row starts, in flight from here
    if (wbase + stride < g.n) load_pass(wbase + stride, rn, en31);
    if (full) {
      *reinterpret_cast<uint2*>(s.branch + wbase + p0) = make_uint2(br[0], br[1]);
    } else {
#pragma unroll
      for (int j = 0; j < kMaskLane; ++j)
        if (p0 + j < cnt) s.branch[wbase + p0 + j] = (uint8_t)(br[j >> 2] >> (8 * (j & 3)));
    }
#pragma unroll
    for (int j = 0; j < kMaskLane; ++j)
      if ((br[j >> 2] >> (8 * (j & 3))) & 1u) s.cidx[wbase + p0 + j] = -1;
    unsigned T;                                        // queued reads of this pass
    unsigned k = warp_exclusive(__popc(pend), &T, lane);
#pragma unroll
    for (int j = 0; j < kMaskLane; ++j)
      if ((pend >> j) & 1u) {
        q_row[wib][k] = r[j];
        q_pos[wib][k] = (uint16_t)((p0 + j) | (((two >> j) & 1u) << 8));
        ++k;
      }
    // the pass's eight words of the heads bitmap: lane 4w + l holds bits 8l..8l+7 of word w
    if (g.min_chain <= 1) {                            // uniform
      unsigned x = lone << (8 * (lane & 3));
      x |= __shfl_xor_sync(0xffffffffu, x, 1);
      x |= __shfl_xor_sync(0xffffffffu, x, 2);
      if ((lane & 3) == 0 && kMaskLane * lane < cnt) s.hb_mask[(wbase >> 5) + (lane >> 2)] = x;
      unsigned L;
      unsigned kl = warp_exclusive(__popc(lone), &L, lane);
      if (nl + L > kMaskBuf) {                         // uniform: this pass would overflow the buffer
        warp_flush(&c->n_lone, s.lone, bl, nl, lane);
        nl = 0;
        __syncwarp();
      }
      kl += nl;
#pragma unroll
      for (int j = 0; j < kMaskLane; ++j)
        if ((lone >> j) & 1u) bl[kl++] = (int32_t)(wbase + p0 + j);
      nl += L;
      // a pass lies inside one tile of the heads bitmap (tiles hold 2^13 reads or more)
      if (lane == 0 && L) atomicAdd(&s.hsum_mask[wbase >> s.h_shift], L * ((1ull << kHeadShift) | 1ull));
    } else if (lane < kMaskSpan / 32 && 32 * lane < cnt) {
      s.hb_mask[(wbase >> 5) + lane] = 0u;
    }
    if (nc + T > kMaskBuf) {                           // uniform: the queue could overflow the buffer
      flush_cands(s, bc, nc, warp_reserve(&c->n_cand, nc, lane), lane);
      nc = 0;
    }
    __syncwarp();                                      // queue written; branch bytes ordered before the fix-ups
    for (unsigned j0 = 0; j0 < T; j0 += 32) {          // warp-uniform
      const unsigned jj = j0 + lane;
      bool cand = false;
      int32_t v = 0;
      if (jj < T) {
        const unsigned q = q_pos[wib][jj];
        const int64_t x = q_row[wib][jj];
        const bool two2 = (q >> 8) != 0;
        v = (int32_t)(wbase + (q & 255u));
        const int32_t w0 = g.col[x];
        const int32_t w1 = two2 ? g.col[x + 1] : w0;
        const int c0 = g.code[x] & 1, c1 = two2 ? (g.code[x + 1] & 1) : c0;
        const bool k0 = (int64_t)rp[w0 + 1] - (int64_t)rp[w0] < 3;
        const bool k1 = two2 && (int64_t)rp[w1 + 1] - (int64_t)rp[w1] < 3;
        // two overlaps to reads of degree <= 2, both on one end: a branch
        if (k0 && k1 && c0 == c1) {
          s.branch[v] = 1;
          s.cidx[v] = -1;
          ++nb;
        } else {
          cand = true;
        }
      }
      const unsigned cm = __ballot_sync(0xffffffffu, cand);
      if (cand) bc[nc + __popc(cm & ((1u << lane) - 1u))] = v;
      nc += __popc(cm);
    }
    __syncwarp();                                      // queue and buffers reused next pass
#pragma unroll
    for (int j = 0; j < kMaskLane; ++j) r[j] = rn[j];
    e31 = en31;
  }
  // one reservation per block for the entries the warps still hold
  __syncthreads();
  unsigned oc = 0, ol = 0;
  if (lane == 0) {
    oc = nc ? atomicAdd(&blk_n[0], nc) : 0;
    ol = nl ? atomicAdd(&blk_n[1], nl) : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    blk_base[0] = blk_n[0] ? atomicAdd(&c->n_cand, blk_n[0]) : 0;
    blk_base[1] = blk_n[1] ? atomicAdd(&c->n_lone, blk_n[1]) : 0;
  }
  __syncthreads();
  oc = blk_base[0] + __shfl_sync(0xffffffffu, oc, 0);
  ol = blk_base[1] + __shfl_sync(0xffffffffu, ol, 0);
  flush_cands(s, bc, nc, oc, lane);
  for (unsigned i = lane; i < nl; i += 32) s.lone[ol + i] = bl[i];
  for (int o = 16; o > 0; o >>= 1) nb += __shfl_down_sync(0xffffffffu, nb, o);
  if (lane == 0 && nb) atomicAdd(&c->n_branch, nb);
}

template <typename RP, bool kAligned>
void launch_mask_kernel(const DevGraph& g, const Scratch& s, const LaunchEnv& env) {
  static const int resident = resident_blocks(k_mask<RP, kAligned>);   // a persistent grid
  const long long need = (g.n + (long long)kMaskWarps * kMaskSpan - 1) / ((long long)kMaskWarps * kMaskSpan);
  const int grid = (int)std::max(1LL, std::min(need, (long long)env.num_sms * resident));
  k_mask<RP, kAligned><<<grid, kBlock, 0, env.stream>>>(g, s);
}

// Successor table of L over the candidates (unmasked reads with overlaps),
// in candidate order: succ[c] = (successor of (c,0), successor of (c,1), read
// id); the overlap (v->w) on end E_v is the way out of (v, 1-E_v) and enters
// (w, E_w), whose incoming suffix is suf(v->w). Also lists the sublist starts
// (list heads and sampled reads) and, among them, the list heads. A
// candidate has one or two overlaps: both entries' fields and their reads'
// candidate indexes (-1: a branch read) are loaded before any store. The
// start lists gather in per-warp shared-memory buffers and reach the global
// lists with one reservation per block at the end (a warp flushes early only
// when its buffer runs full); a start learns its sublist id (kept in the
// successor record's last field for (c,0)) when it is written out.
constexpr int kSuccWarps = kBlock / 32;
constexpr int kSuccStarts = 256;    // sublist starts per warp: oriented candidate | list head << 31

// Writes n buffered sublist starts of one warp to rlist[rbase..] with their
// rr records, and the list heads among them to hlist[hbase..].
__device__ __forceinline__ void put_starts(const Scratch& s, const uint32_t* buf, unsigned n, unsigned rbase,
                                           unsigned hbase, int lane) {
  const unsigned lt = (1u << lane) - 1u;
  unsigned h = 0;
  for (unsigned i0 = 0; i0 < n; i0 += 32) {          // warp-uniform
    const unsigned i = i0 + lane;
    bool head = false;
    if (i < n) {
      const uint32_t e = buf[i];
      const int32_t u = (int32_t)(e & 0x7fffffffu);
      head = (e >> 31) != 0;
      s.rlist[rbase + i] = u;
      // a sampled read's two copies are consecutive starts, (c,0) first: its
      // record keeps the first id, for the walks that end there
      if ((u & 1) == 0) s.succ[u >> 1].w = (int32_t)(rbase + i);
    }
    const unsigned hm = __ballot_sync(0xffffffffu, head);
    if (head) s.hlist[hbase + h + __popc(hm & lt)] = (int32_t)(rbase + i);
    h += __popc(hm);
  }
}

__global__ void __launch_bounds__(kBlock) k_succ(DevGraph g, Scratch s, int ruler_log2) {
  pdl_enter();
  __shared__ uint32_t b_start[kSuccWarps][kSuccStarts];
  __shared__ unsigned blk_n[2], blk_base[2];
  Counters* c = s.ctr;
  const long long N = *(volatile unsigned*)&c->n_cand;
  if (threadIdx.x < 2) blk_n[threadIdx.x] = 0;       // read after the first barrier below
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t* const bs = b_start[wib];
  unsigned ns = 0, nh = 0;                           // buffered starts (warp-uniform), and the heads among them
  // the chain stage's heads bitmap starts from the mask stage's words (lone reads)
  // and so do the tile sums of it
  for (long long w = grid_tid(); w < (g.n + 31) / 32; w += grid_threads()) s.hb[w] = s.hb_mask[w];
  for (long long t = grid_tid(); t < s.h_tiles; t += grid_threads()) s.hsum[t] = s.hsum_mask[t];
  const long long Nw = (N + 31) / 32 * 32;           // whole warps iterate together
  for (long long ci = grid_tid(); ci < Nw; ci += grid_threads()) {
    int s0 = -1, s1 = -1;
    bool r0 = false, r1 = false;
    if (ci < N) {
      int32_t v;
      if (link_candidate(g, s, ci, N, s0, s1, v)) {
        reinterpret_cast<int4*>(s.rr)[ci] = make_int4(-1, 0, -1, 0);   // not yet reached by a sublist walk
        const bool smp = sampled(v, ruler_log2) != 0;
        r0 = s1 < 0 || smp;              // (c,0) has no predecessor when (c,1) has no successor
        r1 = s0 < 0 || smp;
      }
    }
    const bool h0 = r0 && s1 < 0, h1 = r1 && s0 < 0;
    const unsigned m0 = __ballot_sync(0xffffffffu, r0), m1 = __ballot_sync(0xffffffffu, r1);
    const unsigned slot = ns + __popc(m0 & lt) + __popc(m1 & lt);
    if (r0) bs[slot] = (uint32_t)(2 * ci) | (h0 ? 0x80000000u : 0u);
    if (r1) bs[slot + (r0 ? 1 : 0)] = (uint32_t)(2 * ci + 1) | (h1 ? 0x80000000u : 0u);
    ns += __popc(m0) + __popc(m1);
    nh += __popc(__ballot_sync(0xffffffffu, h0)) + __popc(__ballot_sync(0xffffffffu, h1));
    __syncwarp();
    if (ns > kSuccStarts - 64) {         // an iteration adds at most 64 starts
      unsigned rb = 0, hb = 0;
      if (lane == 0) { rb = atomicAdd(&c->n_rulers, ns); hb = nh ? atomicAdd(&c->n_hlist, nh) : 0u; }
      put_starts(s, bs, ns, __shfl_sync(0xffffffffu, rb, 0), __shfl_sync(0xffffffffu, hb, 0), lane);
      ns = 0;
      nh = 0;
    }
    __syncwarp();
  }
  // one reservation per block for the starts the warps still hold
  __syncthreads();
  unsigned o[2] = {0, 0};
  if (lane == 0) {
    o[0] = ns ? atomicAdd(&blk_n[0], ns) : 0u;
    o[1] = nh ? atomicAdd(&blk_n[1], nh) : 0u;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    blk_base[0] = blk_n[0] ? atomicAdd(&c->n_rulers, blk_n[0]) : 0u;
    blk_base[1] = blk_n[1] ? atomicAdd(&c->n_hlist, blk_n[1]) : 0u;
  }
  __syncthreads();
  for (int f = 0; f < 2; ++f) o[f] = blk_base[f] + __shfl_sync(0xffffffffu, o[f], 0);
  put_starts(s, bs, ns, o[0], o[1], lane);
}

// One thread per sublist start: walk to the next start or the list end. The
// sublist's record keeps read ids: its smallest read and its last oriented
// read as 2v + o.
__global__ void k_walk(Scratch s, int ruler_log2, int64_t limit) {
  pdl_enter();
  Counters* c = s.ctr;
  const long long R = *(volatile unsigned*)&c->n_rulers;
  for (long long r = grid_tid(); r < R; r += grid_threads()) {
    const int32_t x = s.rlist[r];
    const int4 sv = s.succ[x >> 1];
    int32_t y = x, z = (x & 1) ? sv.y : sv.x, vy = sv.z, mn = sv.z, next = -1;
    int32_t cnt = 0;
    for (;;) {
      s.rr[y] = make_int2((int32_t)r, cnt);
      ++cnt;
      mn = min(mn, vy);
      if (z < 0) break;
      const int4 sz = s.succ[z >> 1];
      if (sampled(sz.z, ruler_log2)) { next = sz.w + (z & 1); break; }   // the sublist z starts
      y = z;
      vy = sz.z;
      z = (z & 1) ? sz.y : sz.x;
      if (cnt > limit) { set_error(s.derr, DERR_KERNEL, K_WALK, y); break; }
    }
    s.rec[r] = make_int4(next, cnt, mn, 2 * vy + (y & 1));
    s.pj[0][r].x = kUnresolved;
  }
}

// One thread per list head, one walk over the list of sublists: each sublist
// gets the reads before it and its list's head (pj[0][r] = (kViaHead, reads
// before r, head, 0)), and the list's head the totals (pj[1][head] = (total
// reads, smallest read, last oriented read, 0)); the finals turn the pair into
// the reads from r to the tail. Longer lists are left to pointer jumping,
// which rewrites every record in the direct form (-1, reads to the tail,
// smallest read, last read) into both buffers, so the finals read that form
// whenever it ran.
constexpr int kViaHead = -3;                  // pj x-field of a sublist the list walk resolved

__global__ void k_listwalk(Scratch s) {
  pdl_enter();
  Counters* c = s.ctr;
  const long long H = *(volatile unsigned*)&c->n_hlist;
  for (long long h = grid_tid(); h < H; h += grid_threads()) {
    const int32_t r0 = s.hlist[h];
    int32_t r = r0, mn = 0x7fffffff, steps = 0, tail = -1;
    long long total = 0;
    bool ok = true;
    for (;;) {
      const int4 rc = s.rec[r];
      s.pj[0][r] = make_int4(kViaHead, (int32_t)min(total, 0x7fffffffll), r0, 0);
      total += rc.y;
      mn = min(mn, rc.z);
      if (rc.x < 0) {
        tail = rc.w;                     // the list's last oriented read
        break;
      }
      if (++steps >= kListWalkMax) { ok = false; break; }
      r = rc.x;
    }
    if (!ok || total > 0x7fffffffll) {
      atomicOr(&c->need_jump, 1u);
      continue;
    }
    s.pj[1][r0] = make_int4((int32_t)total, mn, tail, 0);
  }
}

// Pointer jumping over all sublists (grid-synchronised rounds), only when a
// list walk gave up (very long chains). After it, for a sublist on an open
// list: acc = oriented reads from its start to the list tail, mn = smallest
// read id over that span, tail = the list's last oriented read. Sublists on
// directed cycles keep next >= 0. Returns the buffer that holds the result, or -1
// when a barrier gave up.
__device__ __forceinline__ int jump_lists(const Scratch& s, unsigned team) {
  Counters* c = s.ctr;
  const long long T = (long long)team * blockDim.x;
  unsigned R = *(volatile unsigned*)&c->n_rulers;
  for (long long i = grid_tid(); i < R; i += T) {
    const int4 rc = s.rec[i];
    s.pj[0][i] = make_int4(rc.x, rc.y, rc.z, rc.w);
  }
  int rounds = 1;
  while ((1u << rounds) < R + 1u && rounds < 31) ++rounds;
  ++rounds;
  int cur = 0;
  if (!grid_sync(c, s.derr, team)) return -1;
  for (int r = 0; r < rounds; ++r) {
    int nxt = cur ^ 1;
    unsigned active = 0;
    for (long long i = grid_tid(); i < R; i += T) {
      const int4 a = s.pj[cur][i];
      if (a.x >= 0) {
        const int4 b = s.pj[cur][a.x];
        const long long acc = (long long)a.y + b.y;
        s.pj[nxt][i] = make_int4(b.x, acc > 0x7fffffffll ? 0x7fffffff : (int32_t)acc,   // saturates on cycles
                                 min(a.z, b.z), b.w);
        active |= (b.x >= 0);
      } else {
        s.pj[nxt][i] = make_int4(-1, a.y, a.z, a.w);
      }
    }
    active = __syncthreads_or(active);
    if (threadIdx.x == 0 && active) atomicOr(&c->round_flag[r], 1u);   // zeroed by the stage
    cur = nxt;
    if (!grid_sync(c, s.derr, team)) return -1;
    if (*(volatile unsigned*)&c->round_flag[r] == 0) break;
  }
  return cur;
}

// Per chain candidate: combine its two oriented copies. head(list of (c,0))
// is the reverse of tail(list of (c,1)). The contig starts at the
// smaller-id end read, so (c,0) is the walk orientation when that end heads
// the list of (c,0). Candidates of closed chains (no list head reached them)
// are listed for the cycle kernel; candidates cut off by branch reads got
// their record from the successor kernel. A thread takes two candidates at a
// time and issues each level of their dependent loads (successor records;
// rank records; list records; length and entering overlap) together, before
// any store.
constexpr int kFinalItems = 2;

// A list the list walk gave up on is jumped first, by the same (cooperative) grid:
// a kernel of its own for that, which mostly found nothing to do, and one for the
// closed chains (see k_heads) made the step of a 100 Mb genome 99.1 us, not 92.6.
// The jumping is the work of `team` blocks, or more for many sublists (coop_do).
// Three blocks per SM, 80 registers: with four it spills 32 bytes (500 Mb 11.8 us for
// 10.2, 3.1 Gb 22.9 for 20.8).
__global__ void __launch_bounds__(kBlock, 3) k_final(DevGraph g, Scratch s, unsigned team) {
  pdl_enter();
  Counters* c = s.ctr;
  int fb = 0;
  if (*(volatile unsigned*)&c->need_jump != 0) {   // the same for every block: written by the kernel before
    team = coop_team(team, *(volatile unsigned*)&c->n_rulers);
    fb = coop_do(s.derr, &c->jumped, team, [&] { return jump_lists(s, team); });
    if (fb < 0) return;
  }
  const long long N = *(volatile unsigned*)&c->n_cand;
  const long long n = (N + 31) & ~31ll;
  const int4* pj = s.pj[fb];
  const long long T = grid_threads();
  unsigned heads = 0;                      // contig heads this thread marked
  for (long long k0 = grid_tid(); k0 < n; k0 += kFinalItems * T) {   // warp-uniform trip count
    bool in[kFinalItems];
    int32_t v[kFinalItems];
    int4 r01[kFinalItems], p0[kFinalItems], p1[kFinalItems];
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      const int4 sv = k0 + j * T < N ? s.succ[k0 + j * T] : make_int4(-1, -1, 0, 0);
      in[j] = sv.x >= 0 || sv.y >= 0;      // a chain candidate
      v[j] = sv.z;
    }
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j)   // (sublist, position) of (c,0) and (c,1)
      r01[j] = in[j] ? reinterpret_cast<const int4*>(s.rr)[k0 + j * T] : make_int4(-1, 0, -1, 0);
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      p0[j] = r01[j].x >= 0 ? pj[r01[j].x] : make_int4(0, 0, 0, 0);
      p1[j] = r01[j].z >= 0 ? pj[r01[j].z] : make_int4(0, 0, 0, 0);
    }
    // a sublist resolved by the list walk: its list's totals sit at the head
    // (in the other buffer), and the reads from it to the tail are the total
    // less the reads before it
    int4 t0[kFinalItems], t1[kFinalItems];
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      t0[j] = p0[j].x == kViaHead ? s.pj[fb ^ 1][p0[j].z] : make_int4(0, 0, 0, 0);
      t1[j] = p1[j].x == kViaHead ? s.pj[fb ^ 1][p1[j].z] : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      if (p0[j].x == kViaHead) p0[j] = make_int4(-1, t0[j].x - p0[j].y, t0[j].y, t0[j].z);
      if (p1[j].x == kViaHead) p1[j] = make_int4(-1, t1[j].x - p1[j].y, t1[j].y, t1[j].z);
    }
    bool cyc[kFinalItems], ok[kFinalItems];
    int32_t m[kFinalItems], q[kFinalItems], rk[kFinalItems], o[kFinalItems], L[kFinalItems], sin[kFinalItems],
        pout[kFinalItems];
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      cyc[j] = in[j] && (r01[j].x < 0 || r01[j].z < 0 || p0[j].x != -1 || p1[j].x != -1);
      ok[j] = in[j] && !cyc[j];
      const int32_t d0 = p0[j].y - r01[j].y - 1;
      const int32_t d1 = p1[j].y - r01[j].w - 1;
      const int32_t h0 = p1[j].w >> 1, h1 = p0[j].w >> 1;   // first read of the list of (c,0) / (c,1)
      // the smallest read of the chain: (c,0)'s list from c's sublist on and
      // (c,1)'s list (the same reads, reversed) from c's sublist on cover it
      m[j] = min(p0[j].z, p1[j].z);
      q[j] = d0 + d1 + 1;
      o[j] = h0 < h1 ? 0 : 1;
      rk[j] = o[j] == 0 ? d1 : d0;
      if (ok[j] && (m[j] < 0 || h0 == h1)) set_error(s.derr, DERR_KERNEL, K_FINAL, v[j]);
      ok[j] = ok[j] && q[j] >= g.min_chain;
    }
    // the piece's inputs: the read's length and its walk copy's overlaps
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      const long long u = 2 * (k0 + j * T) + o[j];
      L[j] = ok[j] ? g.len[v[j]] : 0;
      sin[j] = ok[j] && rk[j] > 0 ? s.sufin[u] : 0;
      pout[j] = ok[j] && g.pre && rk[j] < q[j] - 1 ? s.preout[u] : 0;
    }
#pragma unroll
    for (int j = 0; j < kFinalItems; ++j) {
      const long long ci = k0 + j * T;
      int32_t reads = 0;                     // of the contig that v heads
      if (ok[j]) {
        int32_t len;
        if (g.pre) {   // x-drop form: l_v[post(e_in) : pre(e_out)], alpha / beta at the contig's ends
          const int32_t first = rk[j] == 0 ? (o[j] == 0 ? 0 : L[j] - 1) : sin[j];
          const int32_t last = rk[j] == q[j] - 1 ? (o[j] == 0 ? L[j] - 1 : 0) : pout[j];
          const int32_t cnt = o[j] == 0 ? last - first + 1 : first - last + 1;
          s.pfirst[ci] = first;
          len = cnt > 0 ? cnt : 0;
        } else {       // the first read whole, each later one the suffix it is entered through
          len = rk[j] == 0 ? L[j] : sin[j];
        }
        s.prd[ci] = make_int4(m[j], rk[j], len, o[j]);
        if (v[j] == m[j]) reads = q[j];
      } else if (in[j] && !cyc[j]) {
        s.prd[ci] = make_int4(-1, -1, 0, 255);
      } else if (!in[j] && ci < N && g.min_chain <= 1) {   // cut off by branch reads: its own contig
        reads = 1;
      }
      mark_heads(s, v[j], reads);
      heads += reads > 0;
      const unsigned slot = warp_append(&c->n_cycle_reads, cyc[j]);
      if (cyc[j]) s.cyc[slot] = (int32_t)ci;
    }
  }
  heads = __reduce_add_sync(0xffffffffu, heads);
  if ((threadIdx.x & 31) == 0 && heads) atomicAdd(&c->n_heads, heads);
}

__global__ void k_cycles(DevGraph g, Scratch s) {
  pdl_enter();
  Counters* c = s.ctr;
  const unsigned C = *(volatile unsigned*)&c->n_cycle_reads;
  if (C == 0 || __syncthreads_or(gave_up(s.derr))) return;
  close_cycles(g, s, C, grid_tid(), grid_threads(), [&] { return grid_sync(c, s.derr, gridDim.x); });
}

// Per-read chain outputs, four consecutive reads per thread: a candidate's record,
// found through its index, or the default (a lone read, when spelled, is its own
// one-read contig). Every read is written once, in order; defaults for all reads
// and then the candidates' records over them, in two kernels, took 18 us by
// events for 1.25M reads, and this takes 13. with_cycles: the closed chains come first, on the same
// (cooperative) grid, by `team` of its blocks or more, when there are any.
__global__ void __launch_bounds__(kBlock, 6) k_export_reads(DevGraph g, Scratch s, bool with_cycles, unsigned team,
                                                         int32_t* cid, int32_t* rank, uint8_t* orient) {
  pdl_enter();
  Counters* c = s.ctr;
  const bool stop = gave_up(s.derr);
  const unsigned C = with_cycles ? *(volatile unsigned*)&c->n_cycle_reads : 0u;   // the same for every block
  if (__syncthreads_or(stop)) return;
  if (C > 0) {
    team = coop_team(team, 2ll * C);
    auto sync = [&] { return grid_sync(c, s.derr, team); };
    if (coop_do(s.derr, &c->closed, team, [&] {
          return close_cycles(g, s, C, grid_tid(), (long long)team * kBlock, sync) && sync() ? 0 : -1;
        }) < 0) return;
  }
  const unsigned N = *(volatile unsigned*)&c->n_cand;
  for (long long v0 = 4 * grid_tid(); v0 < g.n; v0 += 4 * grid_threads()) {
    int64_t row[5];
    int32_t ci[4];
    int4 p[4];
#pragma unroll
    for (int k = 0; k < 5; ++k) row[k] = v0 + k <= g.n ? rowp(g, v0 + k) : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) ci[k] = v0 + k < g.n && row[k + 1] > row[k] ? s.cidx[v0 + k] : -1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool lone = row[k + 1] == row[k] && g.min_chain <= 1;
      p[k] = (unsigned)ci[k] < N ? s.prd[ci[k]] : make_int4(lone ? (int)(v0 + k) : -1, lone ? 0 : -1, 0, lone ? 0 : 255);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (v0 + k >= g.n) break;
      if (cid) cid[v0 + k] = p[k].x;
      if (rank) rank[v0 + k] = p[k].y;
      if (orient) orient[v0 + k] = (uint8_t)p[k].w;
    }
  }
}

__global__ void k_sum_len(DevGraph g, unsigned long long* out) {
  unsigned long long acc = 0;
  for (long long v = grid_tid(); v < g.n; v += grid_threads()) acc += (unsigned long long)g.len[v];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

}  // namespace

int coop_blocks_for_grid_kernels(int num_sms) {
  int a = 0, b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_final, kBlock, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_cycles, kBlock, 0);
  int per = a < b ? a : b;
  if (per > 2) per = 2;
  if (per < 1) per = 1;
  return per * num_sms;
}

cudaError_t launch_validate(const DevGraph& g, DevError* derr, const LaunchEnv& env) {
  k_validate_reads<<<grid_for(g.n, env), kBlock, 0, env.stream>>>(g, derr);
  mark(env, "k_validate_reads");
  k_validate_entries<<<grid_for(g.n, env), kBlock, 0, env.stream>>>(g, derr);
  mark(env, "k_validate_entries");
  return cudaGetLastError();
}

cudaError_t launch_sum_len(const DevGraph& g, unsigned long long* out, const LaunchEnv& env) {
  k_sum_len<<<grid_for(g.n, env), kBlock, 0, env.stream>>>(g, out);
  mark(env, "k_sum_len");
  return cudaGetLastError();
}

cudaError_t launch_mask(const DevGraph& g, const Scratch& s, const LaunchEnv& env) {
  if (s.small) return launch_small(g, s, Tuning{}, kStageMask, nullptr, 0, env, false);
  // the counters and, right behind them, the tile sums of the lone reads
  cudaMemsetAsync(&s.ctr->n_branch, 0,
                  sizeof(Counters) - offsetof(Counters, n_branch) + (size_t)s.h_tiles * sizeof(unsigned long long),
                  env.stream);
  const bool al = (reinterpret_cast<uintptr_t>(g.row_ptr) & 15) == 0;   // 16-byte row_ptr loads
  if (g.rp64) {
    if (al) launch_mask_kernel<int64_t, true>(g, s, env);
    else launch_mask_kernel<int64_t, false>(g, s, env);
  } else {
    if (al) launch_mask_kernel<int32_t, true>(g, s, env);
    else launch_mask_kernel<int32_t, false>(g, s, env);
  }
  mark(env, "k_mask");
  return cudaGetLastError();
}

cudaError_t launch_chains(const DevGraph& g, const Scratch& s, const Tuning& t, const LaunchEnv& env,
                          bool after_mask, bool leave_cycles) {
  if (s.small) return launch_small(g, s, t, kStageChains, nullptr, 0, env, after_mask);
  // restart the chain-stage counters; the head bitmap restarts from the mask
  // stage's words (lone reads; k_succ copies them) and gains the chain heads
  if (!after_mask)
    cudaMemsetAsync(&s.ctr->n_rulers, 0, offsetof(Counters, n_contigs) - offsetof(Counters, n_rulers), env.stream);
  static const int succ_resident = resident_blocks(k_succ);   // persistent grids
  static const int final_resident = resident_blocks(k_final);
  // a persistent grid, but no more blocks than the candidates can use
  const long long N = most_candidates(g);
  auto cap = [&](long long resident_grid, long long items, long long items_per_block) {
    const long long need = (items + items_per_block - 1) / items_per_block;
    return (int)std::max(1LL, std::min(resident_grid, need));
  };
  // k_succ also copies the words of a bitmap of the reads
  cudaError_t e = launch_k(k_succ, cap((long long)env.num_sms * succ_resident, std::max(N, (long long)g.n / 32), kBlock),
                           env, after_mask, g, s, t.ruler_log2);
  if (e != cudaSuccess) return e;
  mark(env, "k_succ");
  e = launch_k(k_walk, grid_for(2 * N, env), env, true, s, t.ruler_log2, (int64_t)(2 * g.n + 1));
  if (e != cudaSuccess) return e;
  mark(env, "k_walk");
  e = launch_k(k_listwalk, grid_for(N, env), env, true, s);   // a list per two oriented candidates, at most
  if (e != cudaSuccess) return e;
  mark(env, "k_listwalk");
  DevGraph gg = g;
  Scratch sc = s;
  unsigned team = (unsigned)env.coop_blocks;
  void* args[] = {&gg, &sc, &team};
  e = coop((const void*)k_final, cap((long long)env.num_sms * final_resident, N, (long long)kBlock * kFinalItems), args,
           env, true);
  if (e != cudaSuccess) return e;
  mark(env, "k_final");
  if (leave_cycles) return cudaGetLastError();
  e = coop((const void*)k_cycles, cap(env.coop_blocks, 2 * N, kBlock), args, env, true);
  if (e != cudaSuccess) return e;
  mark(env, "k_cycles");
  return cudaGetLastError();
}

cudaError_t launch_export_reads(const DevGraph& g, const Scratch& s, int32_t* cid, int32_t* rank, uint8_t* orient,
                                const LaunchEnv& env, bool after_chains) {
  static const int resident = resident_blocks(k_export_reads);
  const long long need = (g.n + 4 * kBlock - 1) / (4 * kBlock);
  bool with_cycles = after_chains && !s.small;
  // as many blocks as the reads or, two per SM, the closed chains can use
  const long long team_need =
      with_cycles ? std::min((2 * most_candidates(g) + kBlock - 1) / kBlock, (long long)env.coop_blocks) : 1;
  const int grid = (int)std::min(std::max(need, team_need), (long long)env.num_sms * resident);
  DevGraph gg = g;
  Scratch sc = s;
  unsigned team = (unsigned)env.coop_blocks;
  void* args[] = {&gg, &sc, &with_cycles, &team, &cid, &rank, &orient};
  cudaError_t e = with_cycles ? coop((const void*)k_export_reads, grid, args, env, true)
                              : launch_k(k_export_reads, grid, env, after_chains, g, s, with_cycles, team, cid, rank,
                                         orient);
  if (e != cudaSuccess) return e;
  mark(env, "k_export_reads");
  return cudaGetLastError();
}

}  // namespace cg
