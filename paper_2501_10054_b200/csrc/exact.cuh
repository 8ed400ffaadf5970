// Access to the packed predictor codes (2, 3, 4 or 8 bits each).
#pragma once
#include <stdint.h>

namespace tardis {

// Code of channel k in a row of packed codes: the row is one bit stream, channel order ascending, lowest bits first (code k
// holds bits [k bits, (k + 1) bits) of it).  With 2, 4 or 8 bits a code never leaves its 32-bit word; a 3-bit code may.
__device__ __forceinline__ uint32_t stream_code(const uint32_t* __restrict__ row, int k, int bits) {
  const int pos = k * bits, w = pos >> 5, sh = pos & 31;
  uint32_t v = row[w] >> sh;
  if (sh + bits > 32) v |= row[w + 1] << (32 - sh);
  return v & ((1u << bits) - 1u);
}

}  // namespace tardis
