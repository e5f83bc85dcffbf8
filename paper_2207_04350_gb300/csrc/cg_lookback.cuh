// cg_lookback.cuh - single-pass exclusive scan over 64-bit values with
// decoupled look-back (sm_103a), shared by the kernels that lay out outputs.
// Tiles take tickets in order, publish their aggregate, then look back over
// their predecessors with the whole block (256 descriptors at a time) until an
// inclusive prefix is found. The wait on a predecessor is bounded; on timeout
// the kernel records DERR_TIMEOUT, and every tile that waits gives up with it.
#pragma once

#include <cuda_runtime.h>

#include "cg_internal.cuh"

namespace cg {

namespace {

constexpr int kItems = 8;                       // items per thread
constexpr int kTileItems = kItems * kBlock;     // 2048 items per tile
constexpr unsigned long long kAgg = 1ull << 62, kPre = 2ull << 62, kValMask = (1ull << 62) - 1;
constexpr long long kLookbackSpins = 1ll << 20;

__device__ __forceinline__ unsigned long long ld_volatile(const unsigned long long* p) {
  return *(const volatile unsigned long long*)p;
}

// All threads of the block: publish this tile's aggregate, find its exclusive
// prefix, publish the inclusive prefix. Returns the exclusive prefix. The block
// looks at 256 predecessors at once, so that a scan whose tiles all run at the
// same time mostly takes one look after the last of them has published; one
// warp looking at 32 at a time follows a chain of prefixes instead.
__device__ unsigned long long lookback(unsigned long long* state, long long tile, unsigned long long agg,
                                       DevError* derr, int where) {
  __shared__ int near_pre[kBlock / 32], near_none[kBlock / 32];   // nearest prefix, nearest unpublished
  __shared__ unsigned long long part[kBlock / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tile == 0) {
    if (tid == 0) atomicExch(&state[0], kPre | agg);
    return 0;
  }
  if (tid == 0) atomicExch(&state[tile], kAgg | agg);
  unsigned long long excl = 0;
  long long base = tile - 1;
  long long spins = 0;
  for (;;) {                                               // block-uniform
    const long long idx = base - tid;
    const unsigned long long w = idx >= 0 ? ld_volatile(&state[idx]) : kPre;   // before tile 0: prefix 0
    const unsigned st = (unsigned)(w >> 62);
    const unsigned pm = __ballot_sync(0xffffffffu, st == 2), nm = __ballot_sync(0xffffffffu, st == 0);
    if (lane == 0) {
      near_pre[warp] = pm ? 32 * warp + __ffs(pm) - 1 : kBlock;
      near_none[warp] = nm ? 32 * warp + __ffs(nm) - 1 : kBlock;
    }
    __syncthreads();
    int first = kBlock, none = kBlock;
#pragma unroll
    for (int k = 0; k < kBlock / 32; ++k) {
      first = min(first, near_pre[k]);
      none = min(none, near_none[k]);
    }
    if (none < first) {                                    // a tile before the nearest prefix has not published yet
      ++spins;
      if (__syncthreads_or(tid == 0 && (spins > kLookbackSpins || ((spins & 63) == 0 && gave_up(derr))))) {
        if (tid == 0) set_error(derr, DERR_TIMEOUT, where, tile);
        return excl;
      }
      __nanosleep(spins < 32 ? 20 : 200);
      continue;                                            // near_pre and near_none are written again
    }
    unsigned long long v = tid <= first ? (w & kValMask) : 0ull;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) part[warp] = v;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kBlock / 32; ++k) excl += part[k];
    if (first < kBlock) break;
    base -= kBlock;
  }
  if (tid == 0) atomicExch(&state[tile], kPre | (excl + agg));
  return excl;
}

// Generic single-pass exclusive scan of `count` 64-bit values.
//   Load:  unsigned long long operator()(long long i)
//   Store: void item(long long i, unsigned long long exclusive)
//          void last(long long count, unsigned long long total)
// Blocks loop over tiles by ticket (state[ticket_index], zero before the
// scan), so every tile a block waits for was taken earlier by a block that is
// already running, whatever the grid and however many blocks the GPU runs at
// once (a GPU shared with other work included).
template <class Load, class Store>
__global__ void __launch_bounds__(kBlock) k_scan(Load ld, Store st, long long count, unsigned long long* state,
                                                 long long ticket_index, DevError* derr, int where) {
  pdl_enter();
  __shared__ unsigned long long sm[kTileItems];
  __shared__ unsigned long long warp_tot[kBlock / 32];
  __shared__ long long s_tile;
  const long long tiles = (count + kTileItems - 1) / kTileItems;
  if ((long long)blockIdx.x >= tiles) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (;;) {
    if (tid == 0) s_tile = (long long)atomicAdd(&state[ticket_index], 1ull);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= tiles) return;                       // block-uniform
    const long long base = tile * kTileItems;
    for (int k = 0; k < kItems; ++k) {
      long long i = base + k * kBlock + tid;
      sm[k * kBlock + tid] = i < count ? ld(i) : 0ull;
    }
    __syncthreads();
    unsigned long long v[kItems], sum = 0;
    for (int k = 0; k < kItems; ++k) { v[k] = sm[tid * kItems + k]; sum += v[k]; }
    unsigned long long inc = sum;
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    unsigned long long warp_excl = 0, agg = 0;
    for (int w = 0; w < kBlock / 32; ++w) {
      if (w < warp) warp_excl += warp_tot[w];
      agg += warp_tot[w];
    }
    unsigned long long run = lookback(state, tile, agg, derr, where) + warp_excl + inc - sum;
    for (int k = 0; k < kItems; ++k) { sm[tid * kItems + k] = run; run += v[k]; }
    __syncthreads();
    for (int k = 0; k < kItems; ++k) {
      long long i = base + k * kBlock + tid;
      if (i < count) {
        unsigned long long e = sm[k * kBlock + tid];
        // the total before the item's store: a store may reuse its load's inputs
        const unsigned long long tot = i == count - 1 ? e + ld(i) : 0ull;
        st.item(i, e);
        if (i == count - 1) st.last(count, tot);
      }
    }
    __syncthreads();                                 // sm and s_tile are reused by the next tile
  }
}

}  // namespace

// Grid of a scan over at most `tiles` tiles: blocks loop over tiles by
// ticket, so the grid need not exceed what runs at once (every scan here fits
// three blocks per SM: at most 80 registers per thread and 16.5 KB of shared
// memory per block).
inline unsigned scan_grid(long long tiles, const LaunchEnv& env) {
  const long long cap = (long long)env.num_sms * 3;
  return (unsigned)(tiles < 1 ? 1 : (tiles < cap ? tiles : cap));
}

}  // namespace cg
