// cg_reduce.cu - TransitiveReduction (Alg. 1: S <- TransitiveReduction(R);
// Sec. 2) on sm_103a: the string graph of an overlap graph.
//
// An entry x = (u->w) is transitive when some read v gives a valid walk
// u -> v -> w that leaves u through x's end of u, passes through v (entered
// through one end, left through the other) and enters w through x's end of w,
// and whose suffixes add up to x's within a tolerance. A pair of reads keeps
// both entries only when neither is transitive.
//
// Rows hold a few entries and most reads none, so the rows with entries are
// listed first, long ones in pieces, and the list is cut into batches of about as
// many entries. Every row's entries are copied in two runs, those that leave
// the read through its 5' end and those that leave through the other, each packed
// into eight bytes. Then a block takes a batch of the list, stages it in
// shared memory and gives every entry (u->v) a thread, which walks the run of
// v's row that leaves v through the other end: every entry of it is a walk u ->
// v -> w, whose w is looked up in u's staged row (in memory when u's row is listed
// in pieces). Everything after that is per
// entry: an entry is kept when neither it nor its mirror is transitive; the kept
// entries are bits of one map over all entries with the count of those before
// each word, and since entries lie in row order that count places both the kept
// entries and the new row offsets.
//
// Where the scratch for that does not fit the memory there is, the same kernels run
// without the records and the two runs (kLean): the walks then read the graph's own
// arrays, every entry of v's row, and need 8 bytes per read with entries and 5.4 per
// entry in place of 16 per read, 16 per read with entries and 13.4 per entry. The call
// on the 3.1 Gb overlap graph takes 374 us so (k_tr_rows 242) and 292 with them.
//
// Nothing waits for the host in between: an invalid graph sets the error word,
// and every later kernel reads it first and returns. The kernels that follow
// an entry to another row run only once all row offsets have passed.
#include <cuda_runtime.h>

#include <algorithm>

#include "cg_internal.cuh"
#include "cg_search.h"

namespace cg {

namespace {

constexpr int kTrTile = 2048;        // entries of one tile of the map: 64 words
constexpr int kTrRows = 4;           // consecutive rows per thread of the row pass
// The list of rows. A row of more than kTrPiece entries is listed as pieces of that
// many, so that any piece fits the staging of a batch behind others. A piece weighs
// its entries, kTrFloor at least: a batch is a run of the list of kTrPackUnits or
// kTrWalkUnits units of weight, from the first piece that starts in it on, which
// bounds both its entries and its pieces however long the rows are and whichever lie
// side by side. Batches of so many rows as hold 960 or 720 entries on average, with
// rows past the staging counted and searched in place by their block, took as long on
// the 3.1 Gb graph; with a row of 10,000 / 50,000 entries among 200 thousand of 8
// k_tr_pack took 4.1 / 103 ms (40 / 48 us now), and with 1,000 rows of 999 side by
// side k_tr_rows 97 ms (5.4). With a floor of 8 a batch holds 6% fewer of the 3.1 Gb
// graph's entries: 53.5 and 143 us for 51.5 and 141.
constexpr int kTrPiece = 768;
constexpr int kTrUnitLog2 = 7;       // a unit: 2^7 half weights, 256 entries
constexpr int kTrPackUnits = 4;      // just under four entries per thread
constexpr int kTrWalkUnits = 3;      // three: the less shared memory the blocks of an SM hold, the more cache the random rows have
constexpr int kTrFloor = 6;          // entries that a piece counts as, at least
constexpr int most_pieces(int units) { return ((units << kTrUnitLog2) - 1) / ((kTrFloor + 1) / 2) + 1; }
constexpr int kTrPackRows = most_pieces(kTrPackUnits), kTrWalkRows = most_pieces(kTrWalkUnits);   // pieces of a batch, at most
constexpr int kTrStage = 2048;       // entries of a batch of the packing, at most
constexpr int kTrHold = 1536;        // of the walks
static_assert((2 * kTrPackUnits << kTrUnitLog2) + kTrPiece <= kTrStage && (2 * kTrWalkUnits << kTrUnitLog2) + kTrPiece <= kTrHold,
              "the units of a batch and a piece that starts in the last");
static_assert(kTrPackRows <= 256 && kTrPackRows <= kBlock && kTrWalkRows <= 128, "find_row's steps, a thread per piece");
constexpr int kTrPart = 1 << 30;     // flag beside the read: a piece of a row in pieces (reads stay below 2^30)
constexpr int kTrHalfBits = 33;      // the list's counter: pieces above, half weights below
constexpr unsigned long long kTrHalves = (1ull << kTrHalfBits) - 1;
constexpr int kTrLocalBits = 20;     // the same of one block of the row pass, 1024 rows of one piece each at most
static_assert(kBlock * kTrRows * (kTrPiece / 2) < 1 << kTrLocalBits && kBlock * kTrRows < 1 << (32 - kTrLocalBits), "");

__device__ __forceinline__ int half_weight(int entries) { return (max(entries, kTrFloor) + 1) >> 1; }

__device__ __forceinline__ bool failed(const DevError* e) { return *(const volatile int*)&e->err != 0; }

// Four consecutive values, by 16-byte loads and stores where `wide`.
template <typename T>
__device__ __forceinline__ void load4(const T* p, long long i, long long n, bool wide, T (&v)[4]) {
  constexpr int kVec = 16 / sizeof(T);
  if (wide && i + 4 <= n) {
#pragma unroll
    for (int k = 0; k < 4; k += kVec) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(p + i + k));
      memcpy(&v[k], &x, 16);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = i + k < n ? p[i + k] : T(0);
  }
}
__device__ __forceinline__ void load4_rows(const DevGraph& g, long long i, bool wide, int64_t (&v)[4]) {
  if (g.rp64) {
    load4(reinterpret_cast<const int64_t*>(g.row_ptr), i, g.n + 1, wide, v);
  } else {
    int32_t w[4];
    load4(reinterpret_cast<const int32_t*>(g.row_ptr), i, g.n + 1, wide, w);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = w[k];
  }
}

// Piece (u, first entry p, z entries) at place `slot` of the list, `half` half weights
// before it; false when it does not fit: there are more pieces than the entries allow,
// in rows that overlap, which the row check finds.
template <bool kLean>
__device__ __forceinline__ bool list_piece(const TrBuffers& t, unsigned slot, unsigned long long half, int u, int p, int z) {
  if (slot >= (unsigned)t.rows_cap) {
    set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, u & ~kTrPart);
    return false;
  }
  if constexpr (kLean) t.lean_rows[slot] = make_int2(u, p);
  else t.rows[slot] = make_int4(u, p, z, 0);
  unsigned unit = (unsigned)(half >> kTrUnitLog2);
  int over = (int)((unsigned)half & ((1u << kTrUnitLog2) - 1u)) + half_weight(z) - (1 << kTrUnitLog2);
  for (; over >= 0; over -= 1 << kTrUnitLog2) {        // units that start in the piece or right behind it
    if (++unit >= (unsigned)t.units_cap) {
      set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, u & ~kTrPart);
      return false;
    }
    t.unit_first[unit] = slot + 1u;
  }
  return true;
}

// A row of more than kTrPiece entries, by one thread, with a reservation of its own.
// Rows without end in an invalid graph are given up as soon as its error is set.
template <bool kLean>
__device__ __forceinline__ void list_long_row(const TrBuffers& t, int u, int a, int z) {
  const int more = (z - 1) / kTrPiece, rest = z - more * kTrPiece;      // whole pieces before the last, its entries
  unsigned long long at =
      atomicAdd(t.listed, ((unsigned long long)(more + 1) << kTrHalfBits) +
                              (unsigned long long)more * (kTrPiece / 2) + (unsigned long long)half_weight(rest));
  for (int i = 0; i <= more; ++i) {
    const int n = i < more ? kTrPiece : rest;
    if (failed(t.derr) || !list_piece<kLean>(t, (unsigned)(at >> kTrHalfBits), at & kTrHalves, u | kTrPart, a + i * kTrPiece, n))
      return;
    at += (1ull << kTrHalfBits) + (unsigned long long)half_weight(n);
  }
}

// Rows: offsets from 0 to m that never decrease, no more entries in a row than
// other reads, every read at least one base long. Lists the rows with entries (read,
// first entry, entries; pieces of long ones), one reservation of places and weight
// per block, and the first piece of every unit of weight, with a record per such read
// and a bit in a map of them.
// Reads every row offset and length once, 12 B per read, four consecutive reads
// per thread by 16-byte loads where the arrays allow.
template <bool kLean>
__global__ void __launch_bounds__(kBlock, 6) k_tr_check(DevGraph g, TrBuffers t, bool wide_rows, bool wide_len) {
  __shared__ unsigned cnt;                             // of the block's rows of one piece: pieces << kTrLocalBits | half weights
  __shared__ unsigned long long base;
  const long long u0 = ((long long)blockIdx.x * kBlock + threadIdx.x) * kTrRows;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  int64_t a[4] = {0, 0, 0, 0};
  int32_t len[4] = {0, 0, 0, 0};
  if (u0 <= g.n) load4_rows(g, u0, wide_rows, a);
  if (u0 < g.n) load4(g.len, u0, g.n, wide_len, len);
  int64_t next = __shfl_down_sync(0xffffffffu, a[0], 1);     // the offset after this thread's last row
  if (lane == 31) next = u0 + 4 <= g.n ? rowp(g, u0 + 4) : 0;
  unsigned full = 0, mine = 0;
#pragma unroll
  for (int k = 0; k < kTrRows; ++k) {
    if (u0 + k >= g.n) continue;
    const int64_t b = k + 1 < kTrRows ? a[k + 1 < kTrRows ? k + 1 : 0] : next;
    if (!row_ok(a[k], b, g.m, g.n, len[k])) {
      set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, u0 + k);
    } else if (b > a[k]) {
      full |= 1u << k;
      if (b - a[k] <= kTrPiece) mine += (1u << kTrLocalBits) + (unsigned)half_weight((int)(b - a[k]));
    }
  }
  // the bits of eight threads make a word of the map
  unsigned bits = full << (4 * (lane & 7));
  for (int o = 1; o < 8; o <<= 1) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
  if ((lane & 7) == 0 && u0 < g.n) t.has[u0 >> 5] = bits;
  unsigned inc = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  unsigned at = 0;
  if (lane == 31 && inc) at = atomicAdd(&cnt, inc);
  at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
  if (u0 == 0) {
    if (a[0] != 0 || rowp(g, g.n) != g.m) set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, -1);
    t.unit_first[0] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0 && cnt)
    base = atomicAdd(t.listed, ((unsigned long long)(cnt >> kTrLocalBits) << kTrHalfBits) + (cnt & ((1u << kTrLocalBits) - 1u)));
  __syncthreads();
  const unsigned slot0 = (unsigned)(base >> kTrHalfBits);
  const unsigned long long half0 = base & kTrHalves;
  for (; full; full &= full - 1) {                     // few threads have more than one row to list
    const int k = __ffs(full) - 1, u = (int)(u0 + k);
    const int first = (int)(k == 0 ? a[0] : k == 1 ? a[1] : k == 2 ? a[2] : a[3]);
    const int z = (int)(k == 0 ? a[1] : k == 1 ? a[2] : k == 2 ? a[3] : next) - first;
    if constexpr (!kLean)
      t.info[u] = make_int4(first, 0, first + z, k == 0 ? len[0] : k == 1 ? len[1] : k == 2 ? len[2] : len[3]);
    if (z <= kTrPiece) {
      list_piece<kLean>(t, slot0 + (at >> kTrLocalBits), half0 + (at & ((1u << kTrLocalBits) - 1u)), u, first, z);
      at += (1u << kTrLocalBits) + (unsigned)half_weight(z);
    } else {
      list_long_row<kLean>(t, u, first, z);
    }
  }
}

// The list as batches of `units` units of weight: how many, and where one starts.
struct TrList {
  long long pieces, units;
  int per;
  const unsigned* unit_first;
  __device__ TrList(const TrBuffers& t, int units_per_batch) : per(units_per_batch), unit_first(t.unit_first) {
    const unsigned long long all = *t.listed;
    pieces = (long long)(all >> kTrHalfBits);
    units = (long long)((all & kTrHalves) >> kTrUnitLog2) + 1;
  }
  __device__ long long batches() const { return (units + per - 1) / per; }
  __device__ long long first(long long batch) const {
    return batch * per < units ? (long long)unit_first[batch * per] : pieces;
  }
};

// A batch, pieces [r0, r1) of the list: their records and the places of their
// entries in the batch, row[j].w the first of piece j. Returns the number of
// entries; *parts: there are pieces of rows in pieces among them. Whole block.
template <int kRows, bool kLean>
__device__ __forceinline__ int load_batch(const DevGraph& g, const TrBuffers& t, long long r0, long long r1, int4* row,
                                          int* warp_tot, bool* parts) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int4 mine = make_int4(0, 0, 0, 0);
  if (r0 + tid < r1) {                                 // at most kRows of them
    if constexpr (kLean) {
      const int2 r = t.lean_rows[r0 + tid];
      mine = make_int4(r.x, r.y, min((int)rowp(g, (r.x & ~kTrPart) + 1) - r.y, kTrPiece), 0);
    } else {
      mine = t.rows[r0 + tid];
    }
  }
  int inc = mine.z;
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  int total = 0;
  mine.w = inc - mine.z;
  for (int w = 0; w < (kRows + 31) / 32; ++w) {
    if (w < warp) mine.w += warp_tot[w];
    total += warp_tot[w];
  }
  if (tid < kRows) row[tid] = mine;
  *parts = __syncthreads_or(mine.x & kTrPart) != 0;
  return total;
}

// The piece of the batch's entry i (places past the last piece start at the batch's
// end).
template <int kRows>
__device__ __forceinline__ int find_row(const int4* row, int i) {
  int j = 0;
#pragma unroll
  for (int step = kRows > 128 ? 128 : 64; step > 0; step >>= 1)
    if (((kRows & (kRows - 1)) == 0 || j + step < kRows) && row[j + step].w <= i) j += step;
  return j;
}

// A read with entries: its first one, the first of the second run (0 when there are no
// runs), the end, the read's length.
template <bool kLean>
__device__ __forceinline__ int4 row_info(const DevGraph& g, const TrBuffers& t, int v) {
  if constexpr (kLean) return make_int4((int)rowp(g, v), 0, (int)rowp(g, v + 1), g.len[v]);
  else return t.info[v];
}

// Entries: columns in range, increasing in the row, not the row's own read and a
// read with entries; codes 0..3. Copies every row in two runs by the end its
// entries leave through, each run in the row's order: 9 B read and 12 written per
// entry. An entry's place in its run is the count of entries of that end before
// it, from the ballots of the block's entries; a piece of a long row adds those
// of the rest of the row, counted by its block, a byte an entry. Its loads wait on one another (row,
// code, column), so that warps hide them: with eight blocks on an SM, at 32
// registers, 51 us for 3.36M entries, with six 56; batches of 720 and 480 entries
// 53 and 56.
template <bool kLean>
__global__ void __launch_bounds__(kBlock, 8) k_tr_pack(DevGraph g, TrBuffers t) {
  pdl_enter();
  __shared__ int4 row[kTrPackRows];
  __shared__ unsigned zeros[kTrStage / 32];            // per word of staged entries: entries leaving through end 0
  __shared__ int before[kTrStage / 32 + 1];            // the same before each word
  __shared__ int rest_before[kTrPackRows], rest_all[kTrPackRows];   // pieces of long rows: entries of end 0 before the piece, in the row
  __shared__ int warp_tot[kBlock / 32];
  if (__syncthreads_or(failed(t.derr))) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const TrList list(t, kTrPackUnits);
  for (long long b = blockIdx.x; b < list.batches(); b += gridDim.x) {
    bool parts;
    const int total = load_batch<kTrPackRows, kLean>(g, t, list.first(b), list.first(b + 1), row, warp_tot, &parts);
    if (!kLean && parts) {
      if (tid < kTrPackRows) rest_before[tid] = rest_all[tid] = 0;
      __syncthreads();
      for (int j = 0; j < kTrPackRows; ++j) {             // block-uniform
        if (!(row[j].x & kTrPart)) continue;
        const int4 iu = t.info[row[j].x & ~kTrPart];
        unsigned zb = 0, za = 0;
        for (unsigned y = (unsigned)iu.x + tid; y < (unsigned)iu.z; y += kBlock) {
          const unsigned end0 = (g.code[y] & 1u) ^ 1u;
          za += end0;
          zb += y < (unsigned)row[j].y ? end0 : 0u;
        }
        za = __reduce_add_sync(0xffffffffu, za);
        zb = __reduce_add_sync(0xffffffffu, zb);
        if (lane == 0) {
          atomicAdd(&rest_all[j], (int)za);
          atomicAdd(&rest_before[j], (int)zb);
        }
      }
    }
    constexpr int kPer = kLean ? 0 : kTrStage / kBlock;
    unsigned cd[kTrStage / kBlock];                    // this thread's staged entries
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = k * kBlock + tid;
      cd[k] = 4;
      if (i < total) {
        const int j = find_row<kTrPackRows>(row, i);
        cd[k] = g.code[row[j].y + (i - row[j].w)];
      }
      const unsigned z = __ballot_sync(0xffffffffu, i < total && (cd[k] & 1) == 0);
      if (lane == 0) zeros[(k * kBlock + tid) >> 5] = z;
    }
    __syncthreads();
    if (!kLean && tid < 32) {                          // two words per lane
      const int z0 = __popc(zeros[2 * lane]), z1 = __popc(zeros[2 * lane + 1]);
      int inc = z0 + z1;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
      }
      before[2 * lane] = inc - z0 - z1;
      before[2 * lane + 1] = inc - z1;
      if (lane == 31) before[kTrStage / 32] = inc;
    }
    __syncthreads();
    auto zeros_before = [&](int i) {
      return before[i >> 5] + (i < kTrStage ? __popc(zeros[i >> 5] & ((1u << (i & 31)) - 1u)) : 0);
    };
    for (int i = tid; i < total; i += kBlock) {
      const int j = find_row<kTrPackRows>(row, i);
      const int u = row[j].x & ~kTrPart, n = row[j].z, s0 = row[j].w, x = row[j].y + (i - s0);
      const int32_t w = g.col[x];
      const unsigned c = g.code[x];
      int a = row[j].y;                                // first entry of the row
      int z = 0, nz = 0;                               // entries of end 0 before this one and in the row
      if constexpr (!kLean) {
        z = zeros_before(i) - zeros_before(s0);
        nz = zeros_before(s0 + n) - zeros_before(s0);
      }
      if (row[j].x & kTrPart) {
        a = row_info<kLean>(g, t, u).x;
        if constexpr (!kLean) {
          z += rest_before[j];
          nz = rest_all[j];
        }
        t.trans[x] = (uint8_t)(c << 1);                // the walks only set what they hit, from any block
      }
      const bool ok = w >= 0 && w < g.n && w != u && c <= 3 && (x == a || g.col[x - 1] < w) &&
                      ((t.has[w >> 5] >> (w & 31)) & 1u);
      if (!ok) set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, x);
      if constexpr (!kLean) {
        if (i == s0) t.info[u].y = a + nz;
        const int at = (c & 1) == 0 ? a + z : a + nz + (x - a - z);
        t.ent[at] = make_uint2(((unsigned)w << 2) | (c & 3u), (unsigned)g.suf[x]);
      }
      if (w < u) t.mir[x] = -1;                        // found from the other side, or missing
    }
    __syncthreads();
  }
}

// One entry z = (v->w) of a walk u -> v -> w: whether it makes the entry x of
// u's row that leads to w transitive (codes and suffixes of the three).
__device__ __forceinline__ bool closes(unsigned cx, unsigned cy, unsigned cz, int32_t sx, int32_t sy, int32_t sz,
                                       int fuzz) {
  if (((cx ^ cy) & 1) != 0 || ((cx ^ cz) & 2) != 0) return false;   // the ends of x
  const long long d = (long long)sy + sz - sx;
  return d <= fuzz && d >= -fuzz;
}

// A block per batch of listed rows, a thread per entry y = (u->v): suffix in
// [1, len-1]; from the smaller read's side, the pair's mirrors; and the entries
// of u's row that a walk through v makes transitive. The look-ups are binary
// searches in shared memory, except for the pieces of a long row, which search the
// row in place. What bounds it is the records, runs and columns
// of the rows v, which lie at random (a sector or two each), and issuing the
// searches, in warps whose lanes walk runs of unequal length. 3.36M entries of
// 412 thousand rows, by events: 141 us (178 with the four searches one after
// another; 157 with batches of 960 entries, 2,048 of them staged, and the mirror's
// code read from its row instead of checked where the mirrors' flags are read). A
// thread per entry walking whole rows and searching u's row in memory took 283,
// after 93 for mirrors found by a search of their own; eight lanes per row, four
// rows of a warp in step, took 476, most of its lanes waiting for longer rows; the
// runs of a warp's entries laid end to end, so that no lane waits, 139 to 160 by
// the entries in flight, for as many instructions as without.
template <bool kLean>
__global__ void __launch_bounds__(kBlock, 6) k_tr_rows(DevGraph g, TrBuffers t, int fuzz) {
  pdl_enter();
  __shared__ int4 row[kTrWalkRows];                       // read, first entry, entries, first of the batch's entries
  __shared__ unsigned key[kTrHold];                    // column << 2 | code
  __shared__ int32_t suf[kTrHold];
  __shared__ uint8_t row_of[kTrHold], hit[kTrHold];
  __shared__ int warp_tot[kBlock / 32];
  if (__syncthreads_or(failed(t.derr))) return;
  const int tid = threadIdx.x;
  const TrList list(t, kTrWalkUnits);
  for (long long b = blockIdx.x; b < list.batches(); b += gridDim.x) {
    bool parts;
    const int total = load_batch<kTrWalkRows, kLean>(g, t, list.first(b), list.first(b + 1), row, warp_tot, &parts);
    for (int i = tid; i < total; i += kBlock) {
      const int j = find_row<kTrWalkRows>(row, i);
      const int x = row[j].y + (i - row[j].w);
      key[i] = ((unsigned)g.col[x] << 2) | g.code[x];
      suf[i] = g.suf[x];
      row_of[i] = (uint8_t)j;
      hit[i] = 0;
    }
    __syncthreads();
    for (int i = tid; i < total; i += kBlock) {
      const int j = row_of[i];
      const int u = row[j].x & ~kTrPart, n = row[j].z, s0 = row[j].w, y = row[j].y + (i - s0);
      const bool whole = (row[j].x & kTrPart) == 0;    // u's row is staged whole
      const unsigned e = key[i];
      const int32_t sy = suf[i];
      const int v = (int)(e >> 2);
      const unsigned cy = e & 3u;
      const int4 iv = row_info<kLean>(g, t, v);        // first entry, first of the second run, end, length
      if (sy < 1 || sy > iv.w - 1) set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, y);
      // v is left through its other end: the first run when it was entered through end 1
      // (of a row without runs, the entries that leave through it)
      const unsigned z1 = (unsigned)(!kLean && (cy & 2u) ? iv.y : iv.z);   // unsigned: z + 4 may pass the largest int
      unsigned z = (unsigned)(kLean || (cy & 2u) ? iv.x : iv.y);
      if (u < v) {
        const int32_t back = find_col(g.col, iv.x, iv.z, u);
        if (back >= 0) t.mir[back] = y;
        else set_error(t.derr, DERR_GRAPH, K_TRANSITIVE, y);
        t.mir[y] = back;
      }
      for (; z < z1; z += 4) {
        uint2 q[4];
        bool use[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if constexpr (kLean) {
            const unsigned cz = z + k < z1 ? g.code[z + k] : 0u;
            use[k] = z + k < z1 && ((cz ^ (cy >> 1)) & 1u);
            q[k] = use[k] ? make_uint2(((unsigned)g.col[z + k] << 2) | cz, (unsigned)g.suf[z + k]) : make_uint2(0u, 0u);
          } else {
            use[k] = z + k < z1;
            q[k] = use[k] ? t.ent[z + k] : make_uint2(0u, 0u);
          }
        }
        if (whole) {                                   // the four searches step together
          int lo[4] = {s0, s0, s0, s0};                // the last column <= w, or the first one
          for (int len = n; len > 1;) {
            const int half = len >> 1;
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (key[lo[k] + half] <= (q[k].x | 3u)) lo[k] += half;
            len -= half;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const unsigned kx = key[lo[k]];
            if (use[k] && (kx ^ q[k].x) < 4u && closes(kx, cy, q[k].x, suf[lo[k]], sy, (int32_t)q[k].y, fuzz))
              hit[lo[k]] = 1;
          }
        } else {
          const int4 iu = row_info<kLean>(g, t, u);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (!use[k]) continue;
            const int32_t x = find_col(g.col, iu.x, iu.z, (int32_t)(q[k].x >> 2));
            if (x >= 0 && closes(g.code[x], cy, q[k].x, g.suf[x], sy, (int32_t)q[k].y, fuzz))
              t.trans[x] = (uint8_t)(1u | (g.code[x] << 1));
          }
        }
      }
    }
    __syncthreads();
    for (int i = tid; i < total; i += kBlock) {
      const int j = row_of[i];
      if ((row[j].x & kTrPart) == 0) t.trans[row[j].y + (i - row[j].w)] = (uint8_t)(hit[i] | ((key[i] & 3u) << 1));
    }
    __syncthreads();
  }
}

// Per entry: its mirror must have been found, with the ends of the pair exchanged;
// kept when neither is transitive. A block per tile of the map writes the tile's
// words, the kept entries of the tile before each word, and the tile's count.
__global__ void __launch_bounds__(kBlock) k_tr_keep(long long m, const uint8_t* trans, const int32_t* mir, unsigned* keep,
                                                    unsigned* before, unsigned* tile_cnt, DevError* e) {
  pdl_enter();
  if (__syncthreads_or(failed(e))) return;
  constexpr int kPer = kTrTile / kBlock;
  __shared__ unsigned cnt[kTrTile / 32];
  const long long tile = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long x0 = tile * kTrTile + threadIdx.x;
  uint8_t t[kPer];
  int32_t y[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const long long x = x0 + k * kBlock;
    t[k] = x < m ? trans[x] : 1;
    y[k] = x < m ? mir[x] : 0;
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (y[k] < 0) {                                    // an entry whose pair has no entry back
      set_error(e, DERR_GRAPH, K_TRANSITIVE, x0 + k * kBlock);
      y[k] = 0;
    }
    const uint8_t back = trans[y[k]];
    const bool pair = (back >> 1) == (((t[k] >> 1) & 1) << 1 | t[k] >> 2);   // the two ends, exchanged
    if (x0 + k * kBlock < m && !pair) set_error(e, DERR_GRAPH, K_TRANSITIVE, x0 + k * kBlock);
    t[k] = (t[k] | back) & 1;
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const unsigned bits = __ballot_sync(0xffffffffu, t[k] == 0);
    const int w = k * (kBlock / 32) + warp;
    if (lane == 0) {
      keep[tile * (kTrTile / 32) + w] = bits;
      cnt[w] = __popc(bits);
    }
  }
  __syncthreads();
  if (warp == 0) {
    unsigned c[2], inc;
    c[0] = cnt[2 * lane];
    c[1] = cnt[2 * lane + 1];
    inc = c[0] + c[1];
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    const unsigned ex = inc - c[0] - c[1];
    unsigned* const b = before + tile * (kTrTile / 32) + 2 * lane;
    b[0] = ex;
    b[1] = ex + c[0];
    if (lane == 31) tile_cnt[tile] = inc;
  }
}

// One block: the kept entries before every tile, and all of them in *total.
__global__ void __launch_bounds__(1024) k_tr_tiles(unsigned* tile_cnt, long long tiles, unsigned long long* total,
                                                   const DevError* e) {
  pdl_enter();
  if (failed(e)) return;
  __shared__ unsigned warp_tot[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned run = 0;
  for (long long t0 = 0; t0 < tiles; t0 += 1024) {
    const long long t = t0 + threadIdx.x;
    const unsigned v = t < tiles ? tile_cnt[t] : 0u;
    unsigned inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    unsigned all = 0, lower = 0;
    for (int w = 0; w < 32; ++w) {
      if (w < warp) lower += warp_tot[w];
      all += warp_tot[w];
    }
    if (t < tiles) tile_cnt[t] = run + lower + inc - v;
    run += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = run;
}

// The kept entries before entry p.
__device__ __forceinline__ unsigned kept_before(const TrBuffers& t, int64_t p) {
  return t.tile_cnt[p / kTrTile] + t.before[p >> 5] + __popc(t.keep[p >> 5] & ((1u << (p & 31)) - 1u));
}

// The reduced graph: every kept entry to its place, and every row's offset;
// nothing when the entries do not fit. A thread takes four consecutive rows and
// four consecutive entries at a time, whose words of the map are mostly the same
// one (6.2M rows: 39 us by events, 41 with one of each). Offsets in and out may be loaded and stored by 16 bytes when `wide`.
__global__ void __launch_bounds__(kBlock) k_tr_scatter(DevGraph g, TrBuffers t, long long cap, int64_t* row_ptr,
                                                       int32_t* col, uint8_t* code, int32_t* suf, bool wide) {
  pdl_enter();
  if (failed(t.derr)) return;
  const unsigned long long total = *t.total;
  if ((long long)total > cap) return;
  const long long most = max(((long long)g.n + 4) / 4, ((long long)g.m + 3) / 4);
  for (long long i = grid_tid(); i < most; i += grid_threads()) {
    const long long r = 4 * i;
    int64_t p[4] = {0, 0, 0, 0};
    if (r <= g.n) load4_rows(g, r, wide, p);
    unsigned keep = r < g.m ? (t.keep[r >> 5] >> (r & 31)) & 15u : 0u;   // of entries r .. r + 3
    if (keep) {
      unsigned o = kept_before(t, r);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (!((keep >> k) & 1u)) continue;
        col[o] = g.col[r + k];
        code[o] = g.code[r + k];
        suf[o] = g.suf[r + k];
        ++o;
      }
    }
    if (r > g.n) continue;
    int64_t o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      o[k] = k > 0 && p[k] == p[k - 1] ? o[k - 1] : (p[k] < g.m ? (int64_t)kept_before(t, p[k]) : (int64_t)total);
    if (wide && r + 4 <= g.n + 1) {
      reinterpret_cast<longlong2*>(row_ptr + r)[0] = make_longlong2(o[0], o[1]);
      reinterpret_cast<longlong2*>(row_ptr + r)[1] = make_longlong2(o[2], o[3]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (r + k <= g.n) row_ptr[r + k] = o[k];
    }
  }
}

}  // namespace

long long transitive_tiles(long long m) { return (m + kTrTile - 1) / kTrTile; }
// Pieces: a row gives one more than its whole multiples of kTrPiece. Units: a piece of
// z entries weighs at most z / 2 + 4 halves.
long long transitive_pieces(long long n, long long m) { return std::min(n, m) + m / kTrPiece; }
long long transitive_units(long long n, long long m) {
  return ((m / 2 + 1 + 4 * transitive_pieces(n, m)) >> kTrUnitLog2) + 2;
}

template <bool kLean>
static cudaError_t launch_transitive_walks(const DevGraph& g, int fuzz, const TrBuffers& t, const LaunchEnv& env) {
  const long long blocks = std::max(1ll, ((long long)g.n + kTrRows * kBlock - 1) / (kTrRows * kBlock));
  k_tr_check<kLean><<<(unsigned)blocks, kBlock, 0, env.stream>>>(g, t, (reinterpret_cast<uintptr_t>(g.row_ptr) & 15) == 0,
                                                                 (reinterpret_cast<uintptr_t>(g.len) & 15) == 0);
  mark(env, "k_tr_check");
  if (g.m == 0) return cudaGetLastError();
  static const int pack_resident = resident_blocks(k_tr_pack<kLean>), rows_resident = resident_blocks(k_tr_rows<kLean>);
  // persistent grids; no more batches than units, and one block for a graph that has
  // entries but no reads: the row check has refused it by then
  const long long need = std::max(1ll, t.units_cap);
  cudaError_t e = launch_k(k_tr_pack<kLean>, (int)std::min(need, (long long)env.num_sms * pack_resident), env, true, g, t);
  if (e != cudaSuccess) return e;
  mark(env, "k_tr_pack");
  e = launch_k(k_tr_rows<kLean>, (int)std::min(need, (long long)env.num_sms * rows_resident), env, true, g, t, fuzz);
  if (e != cudaSuccess) return e;
  mark(env, "k_tr_rows");
  return cudaGetLastError();
}

cudaError_t launch_transitive(const DevGraph& g, int fuzz, const TrBuffers& t, const LaunchEnv& env) {
  cudaMemsetAsync(t.total, 0, sizeof(unsigned long long), env.stream);
  cudaMemsetAsync(t.listed, 0, sizeof(unsigned long long), env.stream);
  cudaError_t e = t.lean_rows ? launch_transitive_walks<true>(g, fuzz, t, env) : launch_transitive_walks<false>(g, fuzz, t, env);
  if (e != cudaSuccess || g.m == 0) return e;
  const long long tiles = transitive_tiles(g.m);
  e = launch_k(k_tr_keep, (int)tiles, env, true, (long long)g.m, t.trans, t.mir, t.keep, t.before, t.tile_cnt, t.derr);
  if (e != cudaSuccess) return e;
  mark(env, "k_tr_keep");
  e = launch_kb(k_tr_tiles, 1, 1024, env, true, t.tile_cnt, tiles, t.total, t.derr);
  if (e != cudaSuccess) return e;
  mark(env, "k_tr_tiles");
  return cudaGetLastError();
}

cudaError_t launch_transitive_scatter(const DevGraph& g, const TrBuffers& t, long long cap, int64_t* row_ptr, int32_t* col,
                                      uint8_t* code, int32_t* suf, const LaunchEnv& env, bool chained) {
  const bool wide = ((reinterpret_cast<uintptr_t>(g.row_ptr) | reinterpret_cast<uintptr_t>(row_ptr)) & 15) == 0;
  cudaError_t e = launch_k(k_tr_scatter, grid_for(std::max((long long)g.n + 4, (long long)g.m + 3) / 4, env), env, chained,
                           g, t, cap, row_ptr, col, code, suf, wide);
  if (e != cudaSuccess) return e;
  mark(env, "k_tr_scatter");
  return cudaGetLastError();
}

}  // namespace cg
