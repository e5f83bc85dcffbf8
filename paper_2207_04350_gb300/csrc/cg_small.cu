// cg_small.cu - the mask, chain and offsets stages of a small graph in one
// block (sm_103a).
//
// A small graph's stages cost what their chains of dependent round trips cost,
// not bytes: ten kernels of two to four loads in a row each, with a launch, a
// wait for the kernel before and a look at its counters in front of them, every
// load a trip to L2 since another SM wrote the value. In one block the stages are
// a block barrier apart and read what the SM's own L1 holds, a read's place in a
// list is a block scan instead of an atomic counter, and the chains are ranked by
// pointer jumping over all oriented candidates at once: rounds of two loads that
// mostly hit L1, where the walks of a larger graph follow their longest sublist
// read by read. Everything is written where the other kernels of the library
// expect it. The step of a 1 Mb genome: 43.0 us with ten kernels, 28.0 so. (A
// cluster of 16 such blocks, its barrier between the phases, took 46.5: each
// barrier flushes the stores to L2, and the loads after it go there again.)
#include <cuda_runtime.h>

#include "cg_internal.cuh"
#include "cg_stage.cuh"

namespace cg {

namespace {

constexpr int kThreads = 1024, kWarps = kThreads / 32;
constexpr int kWords = (int)(kSmallReads / 32);          // words of 32 reads, at most
constexpr int kMaskWords = 4;                            // words a warp has in flight
constexpr int kJump = 4;                                 // oriented candidates a thread has in flight

struct Shared {
  unsigned cand[kWords], lone[kWords];                   // per word of reads: candidates, lone reads to spell
  unsigned long long warp[2][kWarps];                    // block scans
  unsigned branch;
};

constexpr unsigned long long kField = (1ull << 21) - 1;  // counts of reads, packed three to a word

__device__ long long mask_stage(const DevGraph& g, const Scratch& s, Shared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)g.n, nw = (n + 31) / 32;
  if (tid == 0) sh.branch = 0;
  __syncthreads();
  unsigned nb = 0;
  for (int l0 = warp; l0 < nw; l0 += kWarps * kMaskWords) {            // warp-uniform
    int row[kMaskWords], d[kMaskWords], w0[kMaskWords], w1[kMaskWords];
    unsigned same = 0;                                   // two overlaps on one end
    bool in[kMaskWords];
#pragma unroll
    for (int k = 0; k < kMaskWords; ++k) {
      const int v = 32 * (l0 + kWarps * k) + lane;
      in[k] = v < n;
      row[k] = in[k] ? (int)rowp(g, v) : 0;
      d[k] = in[k] ? (int)rowp(g, v + 1) - row[k] : 0;
    }
#pragma unroll
    for (int k = 0; k < kMaskWords; ++k) {
      const bool one = d[k] == 1 || d[k] == 2, two = d[k] == 2;
      w0[k] = one ? g.col[row[k]] : 0;
      w1[k] = two ? g.col[row[k] + 1] : w0[k];
      if (two && (g.code[row[k]] & 1) == (g.code[row[k] + 1] & 1)) same |= 1u << k;
    }
#pragma unroll
    for (int k = 0; k < kMaskWords; ++k) {
      const int w = l0 + kWarps * k, v = 32 * w + lane;
      if (w >= nw) break;                                // warp-uniform
      const bool one = d[k] == 1 || d[k] == 2;
      bool branch = d[k] >= 3;
      // two overlaps to reads of degree <= 2, both on one end: a branch
      if (d[k] == 2 && ((same >> k) & 1u))
        branch = rowp(g, w0[k] + 1) - rowp(g, w0[k]) < 3 && rowp(g, w1[k] + 1) - rowp(g, w1[k]) < 3;
      if (in[k]) s.branch[v] = branch;
      if (branch) s.cidx[v] = -1;
      const unsigned cb = __ballot_sync(0xffffffffu, one && !branch);
      const unsigned lb = __ballot_sync(0xffffffffu, in[k] && d[k] <= 0 && g.min_chain <= 1);
      nb += __popc(__ballot_sync(0xffffffffu, branch));
      if (lane == 0) {
        sh.cand[w] = cb;
        sh.lone[w] = lb;
        s.hb_mask[w] = lb;
      }
    }
  }
  if (lane == 0 && nb) atomicAdd(&sh.branch, nb);
  __syncthreads();
  // the lists, in order of the reads: a run of words per thread
  const int per = (nw + kThreads - 1) / kThreads, l0 = tid * per, l1 = min(nw, l0 + per);
  unsigned long long mine = 0;
  for (int l = l0; l < l1; ++l) mine += __popc(sh.cand[l]) + ((unsigned long long)__popc(sh.lone[l]) << 21);
  unsigned long long total;
  const unsigned long long at = block_exclusive<kWarps>(mine, sh.warp[0], &total);
  unsigned ci = (unsigned)(at & kField), li = (unsigned)((at >> 21) & kField);
  for (int l = l0; l < l1; ++l) {
    const int v0 = 32 * l;
    for (unsigned b = sh.cand[l]; b; b &= b - 1, ++ci) {
      const int v = v0 + __ffs(b) - 1;
      s.cand[ci] = v;
      s.cidx[v] = (int32_t)ci;
    }
    for (unsigned b = sh.lone[l]; b; b &= b - 1, ++li) s.lone[li] = v0 + __ffs(b) - 1;
  }
  if (tid == 0) {
    s.ctr->n_cand = (unsigned)(total & kField);
    s.ctr->n_lone = (unsigned)((total >> 21) & kField);
    s.ctr->n_branch = sh.branch;
  }
  return (long long)(total & kField);
}

// N candidates; the lists of the mask stage are visible to all.
__device__ void chain_stage(const DevGraph& g, const Scratch& s, long long N) {
  Counters* c = s.ctr;
  const int tid = threadIdx.x;
  constexpr int kCounters = (int)((offsetof(Counters, n_contigs) - offsetof(Counters, n_rulers)) / 4);
  if (tid < kCounters) (&c->n_rulers)[tid] = 0u;
  for (long long w = tid; w < (g.n + 31) / 32; w += kThreads) s.hb[w] = s.hb_mask[w];
  for (long long ci = tid; ci < N; ci += kThreads) {
    int s0, s1;
    int32_t v;
    link_candidate(g, s, ci, N, s0, s1, v);
    s.pj[0][2 * ci] = make_int4(s0, 1, v, 2 * v);
    s.pj[0][2 * ci + 1] = make_int4(s1, 1, v, 2 * v + 1);
  }
  __syncthreads();
  // pointer jumping: (next, reads from here to the end of the span, smallest
  // read and last oriented read of the span); a round after which no pointer
  // moves any more ends it, and on closed chains the bound on the rounds
  const int M = (int)(2 * N);
  int rounds = 1;
  while ((1ll << rounds) < M + 1 && rounds < 31) ++rounds;
  ++rounds;
  int cur = 0;
  for (int r = 0; r < rounds; ++r) {
    const int4* from = s.pj[cur];
    int4* to = s.pj[cur ^ 1];
    int active = 0;
    for (int u0 = tid; u0 < M; u0 += kJump * kThreads) {
      int4 a[kJump], b[kJump];
#pragma unroll
      for (int k = 0; k < kJump; ++k) a[k] = u0 + k * kThreads < M ? from[u0 + k * kThreads] : make_int4(-1, 0, 0, 0);
#pragma unroll
      for (int k = 0; k < kJump; ++k)
        if (a[k].x >= 0) b[k] = from[a[k].x];
#pragma unroll
      for (int k = 0; k < kJump; ++k) {
        if (a[k].x >= 0) {
          const long long sum = (long long)a[k].y + b[k].y;               // saturates on closed chains
          a[k] = make_int4(b[k].x, sum > 0x7fffffffll ? 0x7fffffff : (int)sum, min(a[k].z, b[k].z), b[k].w);
          active |= b[k].x >= 0;
        }
        if (u0 + k * kThreads < M) to[u0 + k * kThreads] = a[k];
      }
    }
    cur ^= 1;
    if (!__syncthreads_or(active)) break;
  }
  // each candidate's two copies together: head(list of (c,0)) is the reverse of tail(list of (c,1))
  const int4* pj = s.pj[cur];
  int heads = 0;
  for (long long ci = tid; ci < N; ci += kThreads) {
    const int4 sv = s.succ[ci], p0 = pj[2 * ci], p1 = pj[2 * ci + 1];
    const int32_t v = sv.z;
    if (sv.x < 0 && sv.y < 0) {                          // cut off by branch reads: its own contig, or in none
      if (g.min_chain <= 1) {
        mark_head(s, v, 1);
        ++heads;
      }
      continue;
    }
    if (p0.x >= 0 || p1.x >= 0) {                        // on a closed chain
      s.cyc[atomicAdd(&c->n_cycle_reads, 1u)] = (int32_t)ci;
      continue;
    }
    const int32_t d0 = p0.y - 1, d1 = p1.y - 1, h0 = p1.w >> 1, h1 = p0.w >> 1;
    const int32_t m = min(p0.z, p1.z), q = d0 + d1 + 1;
    const int o = h0 < h1 ? 0 : 1;
    const int32_t rk = o == 0 ? d1 : d0;
    if (h0 == h1) set_error(s.derr, DERR_KERNEL, K_FINAL, v);
    if (q >= g.min_chain) {
      s.prd[ci] = make_int4(m, rk, piece_len(g, s, v, (int32_t)ci, (int32_t)(2 * ci + o), rk, q), o);
      if (v == m) {
        mark_head(s, m, q);
        ++heads;
      }
    } else {
      s.prd[ci] = make_int4(-1, -1, 0, 255);
    }
  }
  heads = (int)__reduce_add_sync(0xffffffffu, (unsigned)heads);
  if ((tid & 31) == 0 && heads) atomicAdd(&c->n_heads, (unsigned)heads);
  __syncthreads();
  const unsigned C = *(volatile unsigned*)&c->n_cycle_reads;
  if (C > 0) {
    close_cycles(g, s, C, tid, kThreads, [] {
      __syncthreads();
      return true;
    });
    __syncthreads();
  }
}

__device__ void offsets_stage(const DevGraph& g, const Scratch& s, const PieceStore& ps, Shared& sh) {
  Counters* c = s.ctr;
  const int tid = threadIdx.x;
  // contig index and first walk position of every head: a scan over the words of
  // the heads bitmap, `per` consecutive ones per thread
  const int nw = (int)((g.n + 31) / 32), per = (nw + kThreads - 1) / kThreads;
  unsigned long long mine = 0;
  for (int k = 0; k < per; ++k) {
    const int w = tid * per + k;
    if (w >= nw) break;
    const unsigned bits = s.hb[w], lone = s.hb_mask[w];
    unsigned long long reads = __popc(lone);
    for (unsigned b = bits & ~lone; b; b &= b - 1) reads += (unsigned)s.headq[32 * w + __ffs(b) - 1];
    mine += ((unsigned long long)__popc(bits) << kHeadShift) | reads;
  }
  unsigned long long all;
  unsigned long long e = block_exclusive<kWarps>(mine, sh.warp[1], &all);
  unsigned contigs = (unsigned)(all >> kHeadShift);
  unsigned long long W = all & ((1ull << kHeadShift) - 1);
  if (W > (unsigned long long)g.n) {                     // contigs of more reads than there are: not a string graph
    if (tid == 0) set_error(s.derr, DERR_KERNEL, K_SCAN_HEADS, (long long)W);
    contigs = 0;
    W = 0;
  }
  {
    unsigned k = (unsigned)(e >> kHeadShift);
    unsigned long long r = e & ((1ull << kHeadShift) - 1);
    for (int x = 0; x < per; ++x) {
      const int w = tid * per + x;
      if (w >= nw) break;
      const unsigned lone = s.hb_mask[w];
      s.wp[w] = k;
      for (unsigned b = s.hb[w]; b; b &= b - 1, ++k) {   // contigs in order of their smallest read
        const int i = __ffs(b) - 1;
        const unsigned q = (lone >> i) & 1u ? 1u : (unsigned)s.headq[32 * w + i];
        s.qd[k] = (int32_t)q;
        s.cbase[k] = r;
        r += q;
      }
    }
  }
  if (tid == 0) {
    c->n_contigs = contigs;
    c->n_walk = (unsigned)W;
    s.cbase[contigs] = W;
    if (contigs == 0) {                                  // nothing to scan below
      s.contig_off[0] = 0;
      if (ps.user_off && ps.user_cap >= 1) ps.user_off[0] = 0;
      c->total_bases = 0;
      c->n_tiles = 0;
    }
  }
  if (tid < kTicketSets) s.tickets[kTicketStride * tid] = 0ull;   // for a spelling right after
  __syncthreads();
  scatter_reads(g, s, false, tid, kThreads);
  __syncthreads();
  // piece offsets, four positions per thread at a time
  unsigned long long run = 0;
  for (long long i = 0; i < (long long)W; i += 4 * kThreads) {   // block-uniform
    const long long i0 = i + 4 * tid;
    int32_t L[4], f[4];
    if (i0 + 4 <= (long long)W) {
      const int4 a = *reinterpret_cast<const int4*>(s.wlen + i0), b = *reinterpret_cast<const int4*>(s.wfirst + i0);
      L[0] = a.x; L[1] = a.y; L[2] = a.z; L[3] = a.w;
      f[0] = b.x; f[1] = b.y; f[2] = b.z; f[3] = b.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        L[k] = i0 + k < (long long)W ? s.wlen[i0 + k] : 0;
        f[k] = i0 + k < (long long)W ? s.wfirst[i0 + k] : -1;
      }
    }
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) sum += (unsigned)L[k];
    e = run + block_exclusive<kWarps>(sum, sh.warp[0], &all);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i0 + k >= (long long)W) break;
      ps.item(i0 + k, (long long)e, L[k], f[k]);
      e += (unsigned)L[k];
      if (i0 + k == (long long)W - 1) ps.last((long long)W, e);
    }
    run += all;
    __syncthreads();                                     // sh.warp is written again
  }
}

__global__ void __launch_bounds__(kThreads, 1) k_small(DevGraph g, Scratch s, PieceStore ps, int stages) {
  pdl_enter();
  __shared__ Shared sh;
  long long N = 0;
  if (stages & kStageMask) N = mask_stage(g, s, sh);
  if (stages & kStageChains) {
    if (stages & kStageMask) __syncthreads();
    else N = (long long)*(volatile unsigned*)&s.ctr->n_cand;
    chain_stage(g, s, N);
  }
  if (stages & kStageOffsets) offsets_stage(g, s, ps, sh);
}

}  // namespace

cudaError_t launch_small(const DevGraph& g, const Scratch& s, const Tuning& t, int stages, int64_t* user_off,
                         long long user_cap, const LaunchEnv& env, bool chained) {
  const PieceStore ps{s.out_off, s.contig_off, s.tile_seg, s.tiles_cap, t.tile_bytes, s.ctr, s.derr, user_off, user_cap};
  cudaError_t e = launch_kb(k_small, 1, kThreads, env, chained, g, s, ps, stages);
  if (e != cudaSuccess) return e;
  mark(env, stages == kStageMask ? "k_mask" : stages == kStageChains ? "k_chains" : stages == kStageOffsets ? "k_offsets"
                                                                                                         : "k_small");
  return cudaGetLastError();
}

}  // namespace cg
