// Float32 to float64 without the conversion instruction.
#pragma once

namespace cello {

// A float32 value in float64 by integer instructions: the conversion instruction
// runs at the float64 pipe's rate (1.9 per SM and clock measured), these at 14.
__device__ __forceinline__ double widen(float v) {
  const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)   // normal numbers
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
  return m == 0u ? __hiloint2double((int)u, 0) : (double)v;
}

}  // namespace cello
