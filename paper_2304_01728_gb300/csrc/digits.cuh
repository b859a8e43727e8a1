// Signed digits of fixed-point numbers, exact in bf16 (cells.cuh).
#pragma once
#include "internal.h"

namespace dpgmg {

// the signed 8-bit digits of two fixed-point values (below 127.4 2^48), the leading one
// first, as pairs of bf16: f's in the low halves, g's in the high ones
__device__ __forceinline__ void digit_pairs(long long f, long long g, uint32_t d[DG_S]) {
  const long long bias = 0x0080808080808080ll;
  f += bias;
  g += bias;
  const uint32_t w[4] = {(uint32_t)f, (uint32_t)(f >> 32), (uint32_t)g, (uint32_t)(g >> 32)};
#pragma unroll
  for (int s = 0; s < DG_S; ++s) {
    const int byte = DG_S - 1 - s;   // digit 0 is the leading one
    const uint32_t sel = 0x7650 | (byte & 3);
    const float a = __uint_as_float(__byte_perm(w[byte >> 2], 0x4B000000u, sel)) - 8388736.f;      // - (2^23 + 128)
    const float b = __uint_as_float(__byte_perm(w[2 + (byte >> 2)], 0x4B000000u, sel)) - 8388736.f;
    d[s] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
  }
}

}  // namespace dpgmg
