// cg_serve.h - how much pinned host memory a server asks for, for the server and
// for host code (which tests it).
#pragma once

#include <cstddef>
#include <cstdint>

namespace cg {

constexpr size_t kResultUnit = 65536;            // results are cut from the pinned memory in units of this

// The results that wait to be released are mostly those of the requests within the
// budget, so a server of a small budget, or one of several on a host, locks no more
// than that; a GiB holds what 16 workers of 42 Mb requests have waiting.
inline size_t pinned_result_bytes(uint64_t hbm_budget_bytes) {
  const uint64_t most = uint64_t(1) << 30;
  return (size_t)((hbm_budget_bytes < most ? hbm_budget_bytes : most) / kResultUnit * kResultUnit);
}

}  // namespace cg
