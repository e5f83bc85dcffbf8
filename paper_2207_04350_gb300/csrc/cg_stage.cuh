// cg_stage.cuh - what the kernels of one stage share with the kernel that runs
// all stages of a small graph (cg_small.cu): the work on one candidate or walk
// position, written for any group of threads (sm_103a).
#pragma once

#include <cuda_runtime.h>

#include "cg_internal.cuh"

namespace cg {

namespace {

constexpr long long kSpinLimit = 1ll << 22;   // barrier polls before giving up (~1 s with backoff)

// Software barrier over the first `blocks` blocks of a kernel launched cooperatively
// (all blocks co-resident). Bounded: a block that waits too long records DERR_TIMEOUT
// and gets false, as does every block that still waits then; such a block arrives at
// no further barrier (an arrival of its own would let the others pass one that a block
// still at work has not reached), so its caller returns.
__device__ bool grid_sync(Counters* c, DevError* e, unsigned blocks) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* gen = &c->bar_gen;
    unsigned g0 = *gen;
    __threadfence();
    unsigned arrived = atomicAdd(&c->bar_count, 1u);
    if (arrived == blocks - 1) {
      c->bar_count = 0;
      __threadfence();
      atomicAdd(&c->bar_gen, 1u);
    } else {
      long long spins = 0;
      while (*gen == g0) {
        if (++spins > kSpinLimit || gave_up(e)) {
          set_error(e, DERR_TIMEOUT, K_JUMP, spins);
          ok = 0;
          break;
        }
        __nanosleep(spins < 64 ? 32 : 256);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Work of the first coop_team() blocks that all blocks use: a round of pointer jumping
// costs its barrier, which grows with the blocks in it, until its items do. The team
// returns a value of at least 0, or -1 when a barrier gave up; the others wait for it,
// with the same limit, in a word that the stage zeroes, which they seldom look at (the
// barrier's own words lie beside it). Whole grid; below 0: nothing to use.
__device__ __forceinline__ unsigned coop_team(unsigned least, long long items) {
  return (unsigned)min((long long)gridDim.x, max((long long)least, items / (2 * (long long)blockDim.x)));
}
template <class Work>
__device__ __forceinline__ int coop_do(DevError* e, unsigned* word, unsigned team, Work work) {
  __shared__ int got;
  if (blockIdx.x < team) {
    const int r = work();
    if (r >= 0 && blockIdx.x == 0 && threadIdx.x == 0) {
      __threadfence();
      atomicExch(word, (unsigned)r + 1u);
    }
    return r;
  }
  if (threadIdx.x == 0) {
    long long spins = 0;
    unsigned x;
    while ((x = *(volatile unsigned*)word) == 0u) {
      if (++spins > kSpinLimit / 16 || gave_up(e)) {
        set_error(e, DERR_TIMEOUT, K_JUMP, spins);
        break;
      }
      __nanosleep(4000);
    }
    __threadfence();
    got = (int)x - 1;
  }
  __syncthreads();
  return got;
}

// Read m is the smallest read of a contig of q reads.
__device__ __forceinline__ void mark_head(const Scratch& s, int32_t m, int32_t q) {
  atomicOr(&s.hb[m >> 5], 1u << (m & 31));
  s.headq[m] = q;
  if (!s.small) atomicAdd(&s.hsum[m >> s.h_shift], (1ull << kHeadShift) | (unsigned)q);
}

// The same by a warp, each lane its read m of a contig of q reads or nothing (q = 0).
// Candidates lie in the reads' order but for the blocks', so a warp's heads mostly lie
// in one tile: one addition for them all. With an addition each, 300 thousand reads in
// chains of ten took the final kernel 30 us, not 17: 800 heads to a tile's sum.
__device__ __forceinline__ void mark_heads(const Scratch& s, int32_t m, int32_t q) {
  const unsigned all = 0xffffffffu, any = __ballot_sync(all, q > 0);
  if (any == 0) return;
  const int lane = threadIdx.x & 31, first = __ffs(any) - 1;
  const int tile = q > 0 ? m >> s.h_shift : -1, at = __shfl_sync(all, tile, first);
  const unsigned here = __ballot_sync(all, tile == at);
  const unsigned sum = __reduce_add_sync(all, tile == at ? (unsigned)q : 0u);
  if (q > 0) {
    atomicOr(&s.hb[m >> 5], 1u << (m & 31));
    s.headq[m] = q;
    if (tile != at) atomicAdd(&s.hsum[tile], (1ull << kHeadShift) | (unsigned)q);
    else if (lane == first) atomicAdd(&s.hsum[at], ((unsigned long long)__popc(here) << kHeadShift) | sum);
  }
}

// Candidate ci's successors (s0 of (c,0), s1 of (c,1); -1: none) from its one or
// two overlaps, and what they hand on: the successor record, each successor's
// entering suffix, and the record of a read cut off by branch reads (false
// then). Both entries' fields and their reads' candidate indexes are loaded
// before any store. N: the number of candidates.
__device__ __forceinline__ bool link_candidate(const DevGraph& g, const Scratch& s, long long ci, long long N, int& s0,
                                               int& s1, int32_t& v) {
  s0 = s1 = -1;
  v = s.cand[ci];
  const int64_t a = rowp(g, v);
  const bool two = rowp(g, v + 1) - a == 2;
  const int32_t w0 = g.col[a], w1 = two ? g.col[a + 1] : 0;
  const int cd0 = g.code[a], cd1 = two ? g.code[a + 1] : 0;
  int32_t q0, q1 = 0, p0 = 0, p1 = 0;
  if (g.pre) {
    q0 = g.post[a]; p0 = g.pre[a];
    if (two) { q1 = g.post[a + 1]; p1 = g.pre[a + 1]; }
  } else {
    q0 = g.suf[a];
    if (two) q1 = g.suf[a + 1];
  }
  // a neighbour's candidate index, -1 for a branch read; an entry without its
  // mirror (a graph loaded unvalidated) may reach a read whose index the mask
  // stage never wrote: an out-of-range value counts as a branch read, so the
  // successor and suffix stores below stay inside their arrays
  int32_t c0 = s.cidx[w0], c1 = two ? s.cidx[w1] : -1;
  if ((uint32_t)c0 >= (uint32_t)N) c0 = -1;
  if ((uint32_t)c1 >= (uint32_t)N) c1 = -1;
  const int32_t u0 = 2 * (int32_t)ci;
  if (c0 >= 0) {                     // (v, 1-ev) leaves through end ev
    const int ev = cd0 & 1, to = 2 * c0 + (cd0 >> 1);
    if (ev == 1) s0 = to; else s1 = to;
    s.sufin[to] = q0;
    if (g.pre) s.preout[u0 + 1 - ev] = p0;
  }
  if (c1 >= 0) {
    const int ev = cd1 & 1, to = 2 * c1 + (cd1 >> 1);
    if (ev == 1) s0 = to; else s1 = to;
    s.sufin[to] = q1;
    if (g.pre) s.preout[u0 + 1 - ev] = p1;
  }
  s.succ[ci] = make_int4(s0, s1, v, 0);
  if (s0 < 0 && s1 < 0) {            // every overlap leads to a branch read: spelled alone, or in no contig
    const bool lone = g.min_chain <= 1;
    s.prd[ci] = make_int4(lone ? v : -1, lone ? 0 : -1, lone ? g.len[v] : 0, lone ? 0 : 255);
    if (g.pre) s.pfirst[ci] = 0;   // its contig head is marked by k_final
    return false;
  }
  return true;
}

// x-drop form (Sec. 4.4): read v (candidate ci), walked as oriented
// candidate u at rank rk of a contig of q reads, contributes
// l_v[post(e_in) : pre(e_out)] with alpha (its first base in walk direction)
// for the first read and beta (its last) for the last one; a piece whose end
// comes before its start is empty. Returns the piece's length; its first
// stored base goes to pfirst.
__device__ __forceinline__ int32_t set_piece(const DevGraph& g, const Scratch& s, int32_t v, int32_t ci, int32_t u,
                                             int32_t rk, int32_t q) {
  const int o = u & 1;
  const int32_t L = g.len[v];
  const int32_t first = rk == 0 ? (o == 0 ? 0 : L - 1) : s.sufin[u];
  const int32_t last = rk == q - 1 ? (o == 0 ? L - 1 : 0) : s.preout[u];
  const int32_t cnt = o == 0 ? last - first + 1 : first - last + 1;
  s.pfirst[ci] = first;
  return cnt > 0 ? cnt : 0;
}

// The bases a chain read adds: the first read whole, each later one the
// suffix of the overlap it is entered through (or, in the x-drop form, its
// piece).
__device__ __forceinline__ int32_t piece_len(const DevGraph& g, const Scratch& s, int32_t v, int32_t ci, int32_t u,
                                             int32_t rk, int32_t q) {
  if (g.pre) return set_piece(g, s, v, ci, u, rk, q);
  return rk == 0 ? g.len[v] : s.sufin[u];
}

// Closed chains (rare). Over their oriented candidates: pointer jumping for
// the smallest oriented read 2v + o of each directed cycle, carried with the
// oriented candidate that holds it (the copy holding (m,0) is the walk, m the
// smallest read), then cut the walk before (m,0) and rank by pointer jumping
// again.
// Over `threads` threads of which this is the tid-th; sync() is a barrier over them
// all that makes their writes visible, false when it gave up: then so is the result.
template <class Sync>
__device__ __forceinline__ bool close_cycles(const DevGraph& g, const Scratch& s, unsigned C, long long tid, long long threads,
                             Sync sync) {
  Counters* c = s.ctr;
  long long N = 2ll * C;
  for (long long i = tid; i < N; i += threads) {
    const int32_t ci = s.cyc[i >> 1], u = 2 * ci + (int)(i & 1);
    const int4 sv = s.succ[ci];
    const int32_t z = (u & 1) ? sv.y : sv.x;
    if (z < 0) set_error(s.derr, DERR_KERNEL, K_CYCLE, u);
    s.c_ptr[0][u] = z;
    s.c_val[0][u] = ((long long)(2 * sv.z + (u & 1)) << 32) | (unsigned)u;
  }
  int rounds = 1;
  while ((1ll << rounds) < N + 1 && rounds < 31) ++rounds;
  ++rounds;
  int cur = 0;
  if (!sync()) return false;
  for (int r = 0; r < rounds; ++r) {
    int nxt = cur ^ 1;
    for (long long i = tid; i < N; i += threads) {
      const int32_t u = 2 * s.cyc[i >> 1] + (int)(i & 1);
      const int32_t p = s.c_ptr[cur][u];
      if (p < 0) continue;
      s.c_val[nxt][u] = min(s.c_val[cur][u], s.c_val[cur][p]);
      s.c_ptr[nxt][u] = s.c_ptr[cur][p];
    }
    cur = nxt;
    if (!sync()) return false;
  }
  // cut: on the walk copy, the oriented candidate before the start has no successor
  for (long long i = tid; i < N; i += threads) {
    const int32_t ci = s.cyc[i >> 1], u = 2 * ci + (int)(i & 1);
    const int32_t head = (int32_t)(s.c_val[cur][u] & 0xffffffffll);   // the oriented candidate holding the smallest read
    s.c_head[u] = head;
    if ((head & 1) == 0) {
      const int4 sv = s.succ[ci];
      const int32_t z = (u & 1) ? sv.y : sv.x;
      const int32_t p = (z == head) ? -1 : z;
      s.c_ptr[0][u] = p;
      s.c_val[0][u] = p < 0 ? 0 : 1;
    }
  }
  cur = 0;
  if (!sync()) return false;
  for (int r = 0; r < rounds; ++r) {
    int nxt = cur ^ 1;
    for (long long i = tid; i < N; i += threads) {
      const int32_t u = 2 * s.cyc[i >> 1] + (int)(i & 1);
      if (s.c_head[u] & 1) continue;
      const int32_t p = s.c_ptr[cur][u];
      if (p >= 0) {
        s.c_val[nxt][u] = s.c_val[cur][u] + s.c_val[cur][p];
        s.c_ptr[nxt][u] = s.c_ptr[cur][p];
      } else {
        s.c_val[nxt][u] = s.c_val[cur][u];
        s.c_ptr[nxt][u] = -1;
      }
    }
    cur = nxt;
    if (!sync()) return false;
  }
  for (long long i = tid; i < N; i += threads) {
    const int32_t ci = s.cyc[i >> 1];
    const int32_t u = 2 * ci + (int)(i & 1);
    const int32_t head = s.c_head[u];
    if (head & 1) continue;
    const int32_t L = (int32_t)s.c_val[cur][head] + 1;      // distance from the start to the cut, plus one
    const int32_t rk = L - 1 - (int32_t)s.c_val[cur][u];
    const int32_t m = s.cand[head >> 1];
    const int32_t v = s.cand[ci];
    if (L >= g.min_chain) {
      s.prd[ci] = make_int4(m, rk, piece_len(g, s, v, ci, u, rk, L), u & 1);
      if (rk == 0) {
        mark_head(s, m, L);
        atomicAdd(&c->n_heads, 1u);
      }
    } else {
      s.prd[ci] = make_int4(-1, -1, 0, 255);
    }
    if (rk == 0) atomicAdd(&c->n_cycles, 1u);
  }
  return true;
}

// Block-wide exclusive prefix of one 64-bit value per thread; the sum of all in
// *total. `tot` is shared memory of W words, the block's warps, free again after
// a barrier.
template <int W>
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
  for (int w = 0; w < W; ++w) {
    if (w < warp) before += tot[w];
    all += tot[w];
  }
  *total = all;
  return before + inc - v;
}

// Block-wide sum, the same scratch.
template <int W>
__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long* tot) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) tot[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long all = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) all += tot[w];
  return all;
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

// Every spelled read goes to walk position first(contig) + rank, with the
// stored-base address of its piece (for one part's layout, an empty piece
// when its contig belongs to another part): forward reads add stored bases
// [len-contrib, len), reverse-complement reads the complement of stored
// bases contrib-1 down to 0. The spelled reads are the lone reads of the mask
// stage (each its own contig, whole and forward) and the candidates with a
// contig in their record (chains long enough, and reads cut off by branch
// reads when those are spelled alone). A thread takes two reads at a time and
// issues each level of their dependent loads together, before any store. Nothing
// with `stop` (gave_up).
constexpr int kScatterItems = 2;

__device__ __forceinline__ void scatter_reads(const DevGraph& g, const Scratch& s, bool stop, long long tid,
                                              long long T) {
  Counters* c = s.ctr;
  const long long L1 = *(volatile unsigned*)&c->n_lone, NC = *(volatile unsigned*)&c->n_cand;
  const long long W = *(volatile unsigned*)&c->n_walk;
  const long long total = stop ? 0 : L1 + NC;
  for (long long k0 = tid; k0 < total; k0 += kScatterItems * T) {
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

}  // namespace

}  // namespace cg
