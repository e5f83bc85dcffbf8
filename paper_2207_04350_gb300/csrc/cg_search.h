// cg_search.h - the check of a row of a graph and the search in a sorted one, for
// kernels and for host code (which tests them on bounds that no test graph reaches).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CG_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define CG_HOST_DEVICE inline
#endif

namespace cg {

// Position of column w in the sorted row of entries [a, b), 0 <= a <= b < 2^31, or
// -1. col[i] is read for a <= i < b alone. The middle is taken from the row's
// length: the sum of two entry indices passes the largest int above entry 2^30.
template <class Col>
CG_HOST_DEVICE int32_t find_col(const Col& col, int32_t a, int32_t b, int32_t w) {
  int32_t lo = a, hi = b;
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (col[mid] < w) lo = mid + 1;
    else hi = mid;
  }
  return lo < b && col[lo] == w ? lo : -1;
}

// Whether the row of entries [a, b) of a graph of m entries and n reads can be that
// of a read of `len` bases: offsets in range and in order, at least one base, and no
// more entries than there are other reads. The last keeps what a kernel counts over
// one row far from the largest int, whatever offsets a malformed graph has.
CG_HOST_DEVICE bool row_ok(int64_t a, int64_t b, int64_t m, int64_t n, int32_t len) {
  return a >= 0 && b >= a && b <= m && b - a < n && len >= 1;
}

}  // namespace cg
