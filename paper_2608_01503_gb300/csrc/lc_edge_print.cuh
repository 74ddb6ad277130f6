// lc_edge_print.cuh — the two fingerprints of a stored entry that the
// symmetry check sums.  Plain arithmetic, so host code compiles it too.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lc {

// SplitMix64's output mix (Steele, Lea and Flood, 2014): a bijection.
__host__ __device__ inline unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

struct EdgePrint {
  unsigned long long a, b;
};

// Fingerprints of the undirected edge {lo, hi} of weight w < 2^31.  The edge alone is
// mixed, and the weight enters each fingerprint in its own way:
//   a = fold((mix ^ w phi) K), phi = 2^64 over the golden ratio, K SplitMix64's
//   b = mix (2 w + 1)
// a is a bijection of mix for a given weight and of the weight for a given
// mix, so two entries of one edge with unequal weights always differ in it;
// entries of different edges that agree in a (there are such pairs: 93 bits
// of input) agree in b as any two numbers do.  A weight mixed into the key
// before it is hashed gives both fingerprints the same such pairs if the
// second one is computed from the first.
// Cost: the edge checks of R-MAT scale 21 (62 M entries, bound by their
// instructions) with its objective 544 us with the second fingerprint a
// function of the first, 549 us with these and the check of nnz.
__host__ __device__ inline EdgePrint edge_print(uint32_t lo, uint32_t hi, uint32_t w) {
  const unsigned long long m = mix64(((unsigned long long)lo << 32) | hi);
  const unsigned long long x = (m ^ (unsigned long long)w * 0x9E3779B97F4A7C15ull) * 0xBF58476D1CE4E5B9ull;
  return EdgePrint{x ^ (x >> 32), m * (2u * w + 1u)};  // 32 bits: w < 2^31
}

}  // namespace lc
