// sf_bracket.h - the bracket of a radix search over 32-bit keys, in the kernel
// (rank_step_kernel) and on the host alike.
#pragma once

#include <stdint.h>

#include "sf_host_device.h"

namespace sf {

// The keys from `lo` to `lo + span` that a search has not ruled out, in up to 256
// bins of 2^shift() keys.  Held as a width: the last bin of a bracket that reaches
// up to 2^32 - 1 would end past 32 bits.
struct KeyBracket {
  uint32_t lo, span;

  static SF_HOST_DEVICE KeyBracket between(uint32_t first, uint32_t last) { return {first, last - first}; }
  SF_HOST_DEVICE uint32_t last() const { return lo + span; }
  SF_HOST_DEVICE bool has(uint32_t key) const { return key - lo <= span; }
  SF_HOST_DEVICE int shift() const {
    if (span < 256u) return 0;
#ifdef __CUDA_ARCH__
    return 24 - __clz(static_cast<int>(span));
#else
    return 24 - __builtin_clz(span);
#endif
  }
  // Only the keys of bin `digit`, one that holds a key of the bracket.
  SF_HOST_DEVICE void narrow(uint32_t digit) {
    const int sh = shift();
    const uint32_t below = digit << sh, bin = (1u << sh) - 1u;
    lo += below;
    span = span - below < bin ? span - below : bin;
  }
};

// Every round of a search leaves the width of a bracket eight bits shorter, and one
// more is lost where the key sought was not in the first bracket.
constexpr int kBracketRounds = 32 / 8 + 1;

}  // namespace sf
