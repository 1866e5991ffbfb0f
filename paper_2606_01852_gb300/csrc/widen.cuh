// Widening of results to the output's FP64.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace tn {

// The binary64 value of a binary32 value, exactly, from the two formats' fields with integer
// operations only (this GPU's FP64 pipe is narrow; a conversion per output element would
// bound a one-slice open output): the exponent is rebiased from 127 to 1023 and the 23
// fraction bits move to the top of the 52; subnormal inputs are normalised; zeros and
// infinities keep their sign, and a NaN its sign and payload with the quiet bit set (as an
// IEEE 754 conversion returns a signaling NaN quieted).
__device__ __forceinline__ double f64_of_f32(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint64_t sign = static_cast<uint64_t>(u >> 31) << 63;
  const uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  uint64_t bits;
  if (e == 0xffu) {
    bits = sign | (uint64_t(0x7ff) << 52) | (uint64_t(m) << 29) | (m ? uint64_t(1) << 51 : 0);
  } else if (e != 0u) {
    bits = sign | (uint64_t(e + (1023 - 127)) << 52) | (uint64_t(m) << 29);
  } else if (m == 0u) {
    bits = sign;
  } else {  // m * 2^-149 with the leading one at bit p: exponent p - 149, fraction below it
    const int p = 31 - __clz(static_cast<int>(m));
    bits = sign | (uint64_t(p - 149 + 1023) << 52) | ((uint64_t(m) << (52 - p)) & ((uint64_t(1) << 52) - 1));
  }
  return __longlong_as_double(static_cast<long long>(bits));
}

// The same for a normal number, by its two halves.
__device__ __forceinline__ bool is_normal(float f) {
  return (__float_as_uint(f) & 0x7f800000u) - 0x00800000u < 0x7f000000u;
}
__device__ __forceinline__ double f64_of_normal(float f) {
  const uint32_t u = __float_as_uint(f);
  return __hiloint2double(static_cast<int>((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                          static_cast<int>(u << 29));
}
__device__ __forceinline__ double2 f64_of_f32(float2 v) {
  if (is_normal(v.x) && is_normal(v.y)) return make_double2(f64_of_normal(v.x), f64_of_normal(v.y));
  return make_double2(f64_of_f32(v.x), f64_of_f32(v.y));
}

}  // namespace tn
