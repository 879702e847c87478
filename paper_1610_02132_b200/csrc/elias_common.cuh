// Recursive Elias code (Appendix A.2, Definition A.1) in closed form for integers < 2^16, and
// the MSB-first bit stream the strings S are written to (stream bit t = bit 31 - t % 32 of
// u32 word t / 32).
//
// For k with bit length m the code is P(m) | bin_m(k) | 0, where P(m) is the code of m - 1
// without its final 0: empty for m <= 2, "10"/"11" for m = 3/4, "10" bin_3(m - 1) for
// m = 5..8, "11" bin_4(m - 1) for m = 9..16. Elias(1) is the single bit 0.
#pragma once

#include "qsgd_common.cuh"

namespace qsgd {

__device__ __forceinline__ uint32_t elias_prefix_len(uint32_t m) {
  return (m > 2 ? 2u : 0u) + (m > 4 ? 3u : 0u) + (m > 8 ? 1u : 0u);
}

// Elias(k), right-aligned in the return value; *len receives its length (<= 23).
__device__ __forceinline__ uint32_t elias_code(uint32_t k, uint32_t* len) {
  const uint32_t m = 32u - (uint32_t)__clz((int)k);
  if (m == 1) { *len = 1; return 0u; }
  uint32_t pv = 0;
  if (m > 8) pv = (3u << 4) | (m - 1u);
  else if (m > 4) pv = (2u << 3) | (m - 1u);
  else if (m > 2) pv = m - 1u;
  *len = m + 1u + elias_prefix_len(m);
  return ((pv << m) | k) << 1;
}

}  // namespace qsgd
