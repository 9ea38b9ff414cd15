// float to double without the FP64 pipe.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mka {

// (double)x, exactly, by moving the exponent and mantissa bits: a conversion instruction takes the FP64 pipe for as long
// as an FMA (64 cycles of a warp's scheduler), also where it is predicated off; these few integer operations do not.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
  uint32_t bits = m, bias = m >= 0x7f800000u ? 0x70000000u : 0x38000000u;   // 1023 - 127, or infinity and NaN to their own
  if (m < 0x00800000u) {                          // zero or subnormal: the leading bit to the implicit one's place
    const int s = m ? __clz((int)m) - 8 : 0;
    bits = (m << s) & 0x007fffffu;
    bias = m ? (uint32_t)(897 - s) << 20 : 0u;
  }
  return __hiloint2double((int)((u & 0x80000000u) | ((bits >> 3) + bias)), (int)(bits << 29));
}

template <typename T>
__device__ __forceinline__ T widen_to(float x) {
  if constexpr (sizeof(T) == 8) return widen(x);
  else return x;
}

}  // namespace mka
