// FP32 -> FP64 on the integer pipe.
#pragma once
#include <cstdint>

namespace mpslcc {

// (double)x without the FP64 pipe, which converts at two values a clock and SM
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), e = u & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

}  // namespace mpslcc
