// cg_search.h - the search in a sorted row of a graph, for kernels and for host
// code (which tests it on bounds that no test graph reaches).
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

}  // namespace cg
