// cg_exchange.cu - the read exchange of a run split over ranks that each hold
// only a slice of the reads (the paper's read exchange, Sec. 4.3), on sm_103a.
//
// Every rank lays out the whole graph (mask, chains, offsets) without the
// reads, so every rank knows every piece: its read, its stored range in a
// virtual 2-bit stream (the graph's `off`), and its place in the output. The
// output is cut into equal runs of output tiles, one per rank (the shares of
// cg_emit_share). Rank r owns reads [rf[r], rf[r+1]) and holds their bases in
// a stream of its own layout. For every share p, the pieces of p's range whose
// reads r owns go, in walk order, into r's segment for p: each as the 32-bit
// words covering its stored range in the virtual stream (word W0 = its lowest
// base / 16, through its highest base / 16 + 1), realigned on the way from r's
// own layout, so the receiver needs nothing but the virtual offsets. The
// receiver, its segments laid end to end by source rank (as an all-to-all
// delivers them), moves every piece's source into its buffer and spells its
// share from there.
#include <cuda_runtime.h>

#include <algorithm>

#include "cg_internal.cuh"
#include "cg_lookback.cuh"
#include "cg_stage.cuh"

namespace cg {

namespace {

// The rank r with rf[r] <= v < rf[r + 1].
__device__ __forceinline__ int owner_of(const int64_t* rf, int n, long long v) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rf[mid] <= v) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

struct XPiece {
  long long W0;      // first virtual word sent
  long long words;   // words sent (0 for an empty piece)
};

// Walk position j: words W0 .. hi / 16 + 1 of its stored bases, the spelling's
// two-word windows.
__device__ __forceinline__ XPiece x_piece(const Scratch& s, long long j) {
  const long long L = s.wlen[j];
  const unsigned long long w = s.wsrc[j];
  const long long src = (long long)(w & ~(1ull << 63));
  const int rc = (int)(w >> 63);
  const long long lo = rc ? src - L + 1 : src, hi = rc ? src : src + L - 1;
  XPiece p;
  p.W0 = L > 0 ? lo >> 4 : 0;
  p.words = L > 0 ? (hi >> 4) + 2 - p.W0 : 0;
  return p;
}

// The share of pair i (pairs are the shares' ranges laid end to end).
__device__ __forceinline__ int share_of_pair(const long long* pair0, int n_shares, long long i) {
  int lo = 0, hi = n_shares - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pair0[mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One block, a thread per share: the share's walk range from the tile map, the
// first pair of each range (their number at [n_shares]), and the counts of
// k_x_sizes cleared.
__global__ void __launch_bounds__(kMaxParts) k_x_ranges(Scratch s, XchgArgs x, int tile_bytes) {
  pdl_enter();
  if (gave_up(s.derr)) return;
  __shared__ long long warp_tot[kMaxParts / 32];
  const int p = (int)threadIdx.x, lane = p & 31, warp = p >> 5;
  long long cnt = 0;
  if (p < x.n_shares) {
    const long long total = *(const volatile long long*)&s.ctr->total_bases;
    const long long T = (total + tile_bytes - 1) / tile_bytes;
    const long long t0 = (long long)p * T / x.n_shares, t1 = (long long)(p + 1) * T / x.n_shares;
    long long a = 1, b = 0;                              // empty
    if (t0 < t1) {
      a = s.tile_seg[t0];
      b = s.tile_seg[t1];
    }
    x.range[2 * p] = a;
    x.range[2 * p + 1] = b;
    cnt = max(0ll, b - a + 1);
    x.send_words[p] = 0ull;
    x.recv_words[p] = 0ull;
  }
  long long inc = cnt;
  for (int o = 1; o < 32; o <<= 1) {
    const long long v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  for (int w = 0; w < warp; ++w) inc += warp_tot[w];
  if (p < x.n_shares) {
    x.pair0[p] = inc - cnt;
    if (p == x.n_shares - 1) x.pair0[x.n_shares] = inc;
  }
}

// Words to each share (send) and from each rank (recv): added up per block in
// shared memory, then one addition each (one per warp and key, found by matching
// lanes, took 45 us for 135 thousand pieces into 8 shares). With `mine` also every
// pair's words when this rank owns its read, else 0. A warp's pieces mostly lie
// in one share, which takes one addition for the warp.
__global__ void __launch_bounds__(kBlock) k_x_sizes(Scratch s, XchgArgs x, uint32_t* mine) {
  pdl_enter();
  if (gave_up(s.derr)) return;
  __shared__ unsigned long long send[kMaxParts], recv[kMaxParts];
  __shared__ long long pair0[kMaxParts + 1];
  __shared__ int64_t rf[kMaxParts + 1];
  const int N = x.n_shares, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i <= N; i += kBlock) {
    pair0[i] = x.pair0[i];
    rf[i] = x.rf[i];
    if (i < N) send[i] = recv[i] = 0ull;
  }
  __syncthreads();
  const long long n_pairs = pair0[N], T = grid_threads();
  const long long n_iter = (n_pairs + T - 1) / T * T;  // whole warps iterate together
  for (long long i = grid_tid(); i < n_iter; i += T) {
    int p = -1;
    unsigned long long out = 0;                        // words this rank sends
    if (i < n_pairs) {
      p = share_of_pair(pair0, N, i);
      const long long j = x.range[2 * p] + (i - pair0[p]);
      const long long v = s.wread[j];
      const bool own = v >= rf[x.rank] && v < rf[x.rank + 1];
      if (own || p == x.rank) {
        const unsigned long long words = (unsigned long long)x_piece(s, j).words;
        if (own) out = words;
        if (p == x.rank && words) atomicAdd(&recv[owner_of(rf, N, v)], words);
      }
      if (mine) mine[i] = (uint32_t)out;
    }
    const int p0 = __shfl_sync(0xffffffffu, p, 0);
    if (__all_sync(0xffffffffu, p == p0 || p < 0)) {   // lanes past the last pair add nothing
      for (int o = 16; o > 0; o >>= 1) out += __shfl_down_sync(0xffffffffu, out, o);
      if (lane == 0 && out) atomicAdd(&send[p0], out);
    } else if (out) {
      atomicAdd(&send[p], out);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < N; i += kBlock) {
    if (send[i]) atomicAdd(&x.send_words[i], send[i]);
    if (recv[i]) atomicAdd(&x.recv_words[i], recv[i]);
  }
}

// Scan over all pairs: the words of the pieces this rank owns; every pair gets
// its exclusive prefix, which is its offset in the send buffer, as the segments
// lie end to end in the order of the shares. A pair that holds the first word of
// a chunk of the buffer is that chunk's first pair.
struct XPairLoad {
  const uint32_t* mine;
  __device__ unsigned long long operator()(long long i) const { return mine[i]; }
};
struct XPairStore {
  const uint32_t* mine;
  long long* slot;
  long long* first;
  __device__ void item(long long i, unsigned long long e) const {
    slot[i] = (long long)e;
    const unsigned long long z = e + mine[i];
    for (unsigned long long c = (e + kPackChunk - 1) / kPackChunk; c * kPackChunk < z; ++c) first[c] = i;
  }
  __device__ void last(long long, unsigned long long) const {}
};

__device__ __forceinline__ uint32_t word_checked(const uint32_t* words, const uint8_t* bytes, long long n_bytes,
                                                 long long w) {
  if (w < 0) return 0u;
  if (4 * w + 4 <= n_bytes) return __ldg(words + w);
  uint32_t r = 0;
  for (int b = 0; b < 4; ++b) {
    const long long i = 4 * w + b;
    if (i < n_bytes) r |= (uint32_t)__ldg(bytes + i) << (8 * b);
  }
  return r;
}

// The pairs this rank owns: a piece's virtual words W0 .. W0 + words - 1, each built
// from the rank's own stream (read v's bases start at my_off[v - rf[rank]] there and
// at off[v] in the virtual stream) with one funnel shift; words outside the rank's
// stream read as 0. A warp takes kPackChunk words of the buffer at a time, whatever
// pieces they belong to, from the chunk's first pair on: kPackWords words per lane in
// flight, each lane stepping through the ends of the pieces in shared memory. Bound
// by the chain of loads that finds a piece's source, then by memory: 41 MB packed
// takes 22 us. With eight pairs per warp it took 41: reads of one rank often follow
// one another on a walk, so that an eighth of the warps held all the words (32
// pairs per warp: 92). Chunks of 1,024 words, or eight in flight: no faster.
// The pairs between a rank's own are passed kPackAhead windows of 32 at a time: the
// call of one rank of 1,024, on 240 thousand pairs, takes 149 us so and took 309 a
// window at a time.
constexpr int kPackWords = 4, kPackAhead = 8;

__global__ void __launch_bounds__(kBlock) k_x_pack(DevGraph g, Scratch s, XchgArgs x, const uint8_t* my_packed,
                                                   long long my_bytes, const int64_t* my_off, const uint32_t* mine,
                                                   const long long* slot, const long long* first, uint32_t* send,
                                                   long long n_words) {
  pdl_enter();
  if (gave_up(s.derr)) return;                            // the scan did: slot and first are not whole
  const unsigned full = 0xffffffffu;
  __shared__ long long s_end[kBlock], s_base[kBlock];     // per piece: its end in the buffer, the base that word 0 would start with
  const int lane = threadIdx.x & 31, warp0 = threadIdx.x & ~31;
  const uint32_t* mw = reinterpret_cast<const uint32_t*>(my_packed);
  const long long my_first = x.rf[x.rank], n_pairs = x.pair0[x.n_shares], safe = my_bytes / 4 - 1;
  const long long T = (grid_threads() >> 5) * kPackChunk;
  for (long long a = (grid_tid() >> 5) * kPackChunk; a < n_words; a += T) {   // warp-uniform
    const long long z = min(a + kPackChunk, n_words);
    long long done = a;
    for (long long i0 = first[a / kPackChunk]; done < z && i0 < n_pairs; i0 += 32) {
      long long i = i0 + lane;
      const long long words = i < n_pairs ? (long long)mine[i] : 0ll;
      const long long at = i < n_pairs ? slot[i] : z;
      const bool have = words != 0 && at < z;
      const unsigned own = __ballot_sync(full, have);
      if (own == 0) {                                     // one rank of many owns few pairs: look for the next one
        for (bool found = false; !found && i0 + 32 < n_pairs;) {
          uint32_t next[kPackAhead];
#pragma unroll
          for (int u = 0; u < kPackAhead; ++u) next[u] = i + 32 * (u + 1) < n_pairs ? mine[i + 32 * (u + 1)] : 0u;
#pragma unroll
          for (int u = 0; u < kPackAhead; ++u) {
            if (found) continue;
            found = __any_sync(full, next[u] != 0);
            if (!found) i0 += 32;
          }
          i = i0 + lane;
        }
        continue;
      }
      bool inside = true;
      if (have) {
        const int p = share_of_pair(x.pair0, x.n_shares, i);
        const long long j = x.range[2 * p] + (i - x.pair0[p]);
        const long long v = s.wread[j];
        const long long b = 16 * x_piece(s, j).W0 + my_off[v - my_first] - g.off[v];   // first base in this rank's stream
        const int c = warp0 + __popc(own & ((1u << lane) - 1));
        s_end[c] = at + words;
        s_base[c] = b - 16 * at;
        inside = b >= 0 && (b >> 4) + words <= safe;
      }
      inside = __all_sync(full, inside);
      __syncwarp();
      const long long end = min(z, __shfl_sync(full, at + words, 31 - __clz(own)));
      int c = warp0;
      long long e = s_end[c], f = s_base[c];
      if (inside) {
        for (long long k0 = done + lane; k0 < end; k0 += 32 * kPackWords) {
          uint32_t lo[kPackWords], hi[kPackWords], sh[kPackWords];
#pragma unroll
          for (int u = 0; u < kPackWords; ++u) {
            const long long k = min(k0 + 32 * u, end - 1);
            while (k >= e) {
              e = s_end[++c];
              f = s_base[c];
            }
            const uint32_t* w = mw + ((f >> 4) + k);
            sh[u] = (uint32_t)(2 * (f & 15));
            lo[u] = __ldg(w);
            hi[u] = __ldg(w + 1);
          }
#pragma unroll
          for (int u = 0; u < kPackWords; ++u)
            if (k0 + 32 * u < end) send[k0 + 32 * u] = __funnelshift_r(lo[u], hi[u], sh[u]);
        }
      } else {
        for (long long k = done + lane; k < end; k += 32) {
          while (k >= e) {
            e = s_end[++c];
            f = s_base[c];
          }
          const long long w = (f >> 4) + k;               // floor, also below 0
          send[k] = __funnelshift_r(word_checked(mw, my_packed, my_bytes, w),
                                    word_checked(mw, my_packed, my_bytes, w + 1), (unsigned)(2 * (f & 15)));
        }
      }
      done = end;
      __syncwarp();                                       // s_end and s_base are written again
    }
  }
}

// The receiver: every piece of its range, its source moved into the receive
// buffer (16 bases per word, the piece's phase within its first word kept). The
// blocks of row r scan the range for the words of the pieces whose reads rank r
// holds; r's segment starts after those of the ranks before it. One launch of all
// scans: one per source rank, each waiting for the one before, took 18 us apiece.
__global__ void __launch_bounds__(kBlock) k_x_place(Scratch s, XchgArgs x, unsigned long long* state, long long state_cap) {
  pdl_enter();
  constexpr int kPer = kXchgTile / kBlock;
  __shared__ unsigned long long tot[kBlock / 32];
  __shared__ long long s_tile;
  if (__syncthreads_or(gave_up(s.derr))) return;
  const int who = (int)blockIdx.y, tid = threadIdx.x;
  const long long j0 = x.range[2 * x.rank], count = x.range[2 * x.rank + 1] - j0 + 1;
  const long long tiles = (count + kXchgTile - 1) / kXchgTile;
  if ((long long)blockIdx.x >= tiles) return;
  const int64_t v0 = x.rf[who], v1 = x.rf[who + 1];
  state += (long long)who * (state_cap + 1);
  unsigned long long seg = 0;
  for (int r = tid; r < who; r += kBlock) seg += x.recv_words[r];
  seg = block_sum<kBlock / 32>(seg, tot);
  for (;;) {
    if (tid == 0) s_tile = (long long)atomicAdd(&state[state_cap], 1ull);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= tiles) return;                           // block-uniform
    const long long i0 = tile * kXchgTile + kPer * tid;
    XPiece q[kPer];
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      q[k].words = 0;
      if (i0 + k < count) {
        const long long v = s.wread[j0 + i0 + k];
        if (v >= v0 && v < v1) q[k] = x_piece(s, j0 + i0 + k);
      }
      sum += (unsigned long long)q[k].words;
    }
    unsigned long long all, e = block_exclusive<kBlock / 32>(sum, tot, &all);
    e += seg + lookback(state, tile, all, s.derr, (int)K_SCAN_OFFSETS);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (q[k].words == 0) continue;
      const unsigned long long w = s.wsrc[j0 + i0 + k];
      const long long src = (long long)(w & ~(1ull << 63));
      s.wsrc[j0 + i0 + k] = (unsigned long long)(16 * (long long)e + (src - 16 * q[k].W0)) | (w & (1ull << 63));
      e += (unsigned long long)q[k].words;
    }
    __syncthreads();                                     // s_tile and tot are reused by the next tile
  }
}

}  // namespace

cudaError_t launch_x_sizes(const Scratch& s, const XchgArgs& x, int tile_bytes, long long n, uint32_t* mine,
                           const LaunchEnv& env) {
  k_x_ranges<<<1, std::max(32, (x.n_shares + 31) & ~31), 0, env.stream>>>(s, x, tile_bytes);
  mark(env, "k_x_ranges");
  cudaError_t e = launch_k(k_x_sizes, grid_for(n, env, 4), env, true, s, x, mine);
  if (e != cudaSuccess) return e;
  mark(env, "k_x_sizes");
  return cudaGetLastError();
}

cudaError_t launch_x_pack(const DevGraph& g, const Scratch& s, const XchgArgs& x, const uint8_t* my_packed,
                          long long my_bytes, const int64_t* my_off, const uint32_t* mine, long long* slot,
                          long long* first, unsigned long long* state, long long state_cap, uint32_t* send,
                          long long n_pairs, long long n_words, const LaunchEnv& env) {
  if (n_pairs <= 0 || n_words <= 0) return cudaSuccess;
  const long long tiles = (n_pairs + kTileItems - 1) / kTileItems;
  if (tiles > state_cap) return cudaErrorInvalidValue;
  cudaMemsetAsync(state, 0, (size_t)(state_cap + 1) * sizeof(unsigned long long), env.stream);
  k_scan<<<scan_grid(tiles, env), kBlock, 0, env.stream>>>(XPairLoad{mine}, XPairStore{mine, slot, first}, n_pairs, state,
                                                           state_cap, s.derr, (int)K_SCAN_OFFSETS);
  mark(env, "k_scan_exchange_pairs");
  cudaError_t e = launch_k(k_x_pack, grid_for(32 * ((n_words + kPackChunk - 1) / kPackChunk), env), env, true, g, s, x,
                           my_packed, my_bytes, my_off, mine, (const long long*)slot, (const long long*)first, send,
                           n_words);
  if (e != cudaSuccess) return e;
  mark(env, "k_x_pack");
  return cudaGetLastError();
}

cudaError_t launch_x_place(const Scratch& s, const XchgArgs& x, long long count, unsigned long long* state,
                           long long state_cap, const LaunchEnv& env) {
  if (count <= 0) return cudaSuccess;
  const long long tiles = (count + kXchgTile - 1) / kXchgTile;
  if (tiles > state_cap) return cudaErrorInvalidValue;
  cudaMemsetAsync(state, 0, (size_t)x.n_shares * (size_t)(state_cap + 1) * sizeof(unsigned long long), env.stream);
  k_x_place<<<dim3((unsigned)std::min(tiles, (long long)env.num_sms * 2), (unsigned)x.n_shares), kBlock, 0, env.stream>>>(
      s, x, state, state_cap);
  mark(env, "k_x_place");
  return cudaGetLastError();
}

}  // namespace cg
