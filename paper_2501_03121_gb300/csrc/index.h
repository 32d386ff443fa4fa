// Index arithmetic that the kernels and the host share, in plain C++.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define TVCG_HD __host__ __device__ __forceinline__
#else
#define TVCG_HD inline
#endif

namespace tvcg {

// q / n for a piece index q >= 0 and n >= 1 pieces per row; one 32-bit
// division where both fit.  n can pass 2^32 while q does not: a row of 2^34
// FP32 elements is 2^32 pieces.
TVCG_HD int64_t piece_row(int64_t q, int64_t n) {
  return ((q | n) >> 32) ? q / n : (int64_t)((uint32_t)q / (uint32_t)n);
}

// Whether a count of barrier arrivals `v` has reached `want`, both modulo 2^32
// and less than 2^31 apart.
TVCG_HD bool arrivals_reached(uint32_t v, uint32_t want) { return (int32_t)(v - want) >= 0; }

}  // namespace tvcg
