// bounds.cuh -- range tests of the kernels that also compile as plain C++, so that
// their edges can be checked without a GPU.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BBTC_HD __host__ __device__ __forceinline__
#else
#define BBTC_HD inline
#endif

namespace bbtc {

// Whether the entries [at, at + count) lie inside [0, size), for any `at` (one taken
// from a row pointer that has not been checked yet may be negative or huge).
BBTC_HD bool span_inside(int64_t at, uint32_t count, int64_t size) {
  return at >= 0 && at <= size && (int64_t)count <= size - at;
}

// Whether record base + i lies before `end` (base <= end): positions reach 2^32 - 1,
// where base + i would wrap to the front of the array.
BBTC_HD bool window_holds(uint32_t base, uint32_t i, uint32_t end) { return i < end - base; }

}  // namespace bbtc
