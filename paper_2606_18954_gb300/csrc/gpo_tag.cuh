// Tags of whole calls in the status words (see Status in gpo_internal.cuh).  Host C++ only.
#pragma once
#include <cstdint>

namespace gpo {

// The n-th tag: a bijection of the 48-bit numbers (odd multiplications modulo 2^48 and
// xor-shifts, each of which has an inverse), so that no tag comes twice in 2^48 calls, spread
// so that small integers or text in memory hardly ever look like a recent one.  0 is no tag
// (one n gives it).
inline uint64_t tag_of(uint64_t n) {
  constexpr uint64_t kMask = (1ull << 48) - 1;
  uint64_t z = (n * 0x9E3779B97F4Bull + 0x2545F4914F6Cull) & kMask;
  z = ((z ^ (z >> 27)) * 0x94D049BB1331ull) & kMask;
  z = ((z ^ (z >> 23)) * 0xBF58476D1CE5ull) & kMask;
  return z ^ (z >> 25);
}

}  // namespace gpo
