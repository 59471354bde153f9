// Conversions between float and double on the integer pipe, bit for bit those
// of the FP64 pipe.  GB300 runs its conversion instructions at the FP64 rate
// (2 lanes per SM clock, measured: float -> double 2.0, double -> float 2.0
// per clock, against 103 FFMA), so a vector pass that converts a few values
// per element is bound by them; six to twelve integer instructions take a
// quarter of that time and leave the FP64 pipe to the arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace lgw {

template <class T, class F>
__host__ __device__ __forceinline__ T bits_as(F x) {
  static_assert(sizeof(T) == sizeof(F), "same size");
  T y;
  memcpy(&y, &x, sizeof y);
  return y;
}

// (double)x: the exponent rebiased by 896, the mantissa moved up 29 bits.
// Subnormals, infinities and NaN convert natively.
__host__ __device__ __forceinline__ double f2d(float x) {
  const uint32_t b = bits_as<uint32_t>(x), a = b & 0x7fffffffu;
  if (a - 0x00800000u >= 0x7f000000u && a != 0) return (double)x;
  const uint32_t hi = (b & 0x80000000u) | (a != 0 ? (a >> 3) + 0x38000000u : 0u);
  return bits_as<double>(((uint64_t)hi << 32) | (uint32_t)(b << 29));
}

// Bits of |x| rounded to the nearest float (ties to even), for 2^-126 <= |x|
// < 2^128: the top 32 of the 61 bits below the exponent's rebias, plus the
// rounding carry (which may run into the exponent, as it should).
__host__ __device__ __forceinline__ uint32_t rn_bits(uint32_t ahi, uint32_t lo) {
  const uint32_t f = ((ahi - 0x38000000u) << 3) | (lo >> 29);
  return f + (((lo & 0x1fffffffu) + 0x0fffffffu + (f & 1u)) >> 29);
}

// (float)x, round to nearest even.
__host__ __device__ __forceinline__ float d2f(double x) {
  const uint64_t b = bits_as<uint64_t>(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, a = hi & 0x7fffffffu;
  const uint32_t s = hi & 0x80000000u;
  if ((a | lo) == 0) return bits_as<float>(s);
  // outside 2^-126 .. 2^127 (exponent fields 897 .. 1150): natively
  if (a - 0x38100000u >= 0x0fe00000u) return (float)x;
  return bits_as<float>(s | rn_bits(a, lo));
}

// bf16(x), round to nearest even in one step: the float's upper half, with
// everything below it deciding the rounding.
__host__ __device__ __forceinline__ __nv_bfloat16 d2bf16(double x) {
  const uint64_t b = bits_as<uint64_t>(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, a = hi & 0x7fffffffu;
  uint16_t r = (uint16_t)(hi >> 16 & 0x8000u);
  if ((a | lo) != 0) {
    if (a - 0x38100000u >= 0x0fe00000u) return __double2bfloat16(x);
    const uint32_t f = ((a - 0x38000000u) << 3) | (lo >> 29);
    const uint32_t below = (f & 0xffffu) | ((lo & 0x1fffffffu) != 0 ? 1u : 0u);
    // the sticky bit never makes a tie: below == 0x8000 only if lo's is zero
    r |= (uint16_t)((f >> 16) + ((below + 0x7fffu + (f >> 16 & 1u)) >> 16));
  }
  return bits_as<__nv_bfloat16>(r);
}

// h = (float)x and l = (float)(x - (double)h): what is left below h is an
// integer of at most 29 bits on x's last place, rounded by its conversion and
// scaled by a power of two.
__host__ __device__ __forceinline__ void split_d(double x, float &h, float &l) {
  const uint64_t b = bits_as<uint64_t>(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, a = hi & 0x7fffffffu;
  if ((a | lo) == 0) {
    h = bits_as<float>(hi);
    l = 0.0f;
    return;
  }
  // exponent fields 950 .. 1149: l's scale and h stay normal
  if (a - 0x3b600000u >= 0x0c800000u) {
    h = (float)x;
    l = (float)(x - (double)h);
    return;
  }
  const uint32_t f = ((a - 0x38000000u) << 3) | (lo >> 29), r = lo & 0x1fffffffu;
  const uint32_t up = (r + 0x0fffffffu + (f & 1u)) >> 29;
  const int32_t d = (int32_t)r - (int32_t)(up << 29);
  h = bits_as<float>((hi & 0x80000000u) | (f + up));
  l = (float)((int32_t)hi < 0 ? -d : d) * bits_as<float>(((a >> 20) - 948u) << 23);
}

}  // namespace lgw
