// lc_bin_rule.cuh — the degree of a row and the bin that takes it.  Plain
// arithmetic, so host code compiles it too.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lc {

// Degree bins of the per-vertex kernels (lc_internal.cuh says what each is).
constexpr int kBins = 10;

// Entries of a row [beg, end), at least 0 and at most INT32_MAX.  The bins are
// built while row_ptr is still being checked, so its values may be anything;
// every phase of the binning takes the degree from here, as 32 bits, so that
// what one phase counts in a bin is what another places there.
__host__ __device__ inline int32_t row_degree(int64_t beg, int64_t end) {
  if (end <= beg) return 0;
  const uint64_t d = (uint64_t)end - (uint64_t)beg;
  return d > (uint64_t)INT32_MAX ? INT32_MAX : (int32_t)d;
}

// The bin of a degree: bin k takes max_deg[k - 1] < deg <= max_deg[k].
__host__ __device__ inline int bin_of(const int32_t *max_deg, int32_t deg) {
  int b = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < kBins - 1; ++k) b += deg > max_deg[k] ? 1 : 0;
  return b;
}

}  // namespace lc
