// Conversions between float and double on the integer pipe, bit for bit those
// of the FP64 pipe.  GB300 runs its conversion instructions at the FP64 rate
// (2 lanes per SM clock, measured: float -> double 2.0, double -> float 2.0
// per clock, against 103 FFMA), so a vector pass that converts a few values
// per element is bound by them; six to twelve integer instructions take a
// quarter of that time and leave the FP64 pipe to the arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
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

__host__ __device__ __forceinline__ int clz64(uint64_t u) {   // u != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)u);
#else
  return __builtin_clzll(u);
#endif
}

// (double)t * 2^sh, rounded once to nearest even where the result is normal.
__host__ __device__ __forceinline__ double ll2d_scaled(long long t, int sh) {
  if (t == 0) return 0.0;
  uint64_t u = t < 0 ? 0ULL - (uint64_t)t : (uint64_t)t;
  const int lz = clz64(u);
  u <<= lz;
  const uint32_t below = (uint32_t)u & 0x7ffu;
  u >>= 11;   // 53 bits, the leading one at 2^52
  u += (below + 0x3ffu + ((uint32_t)u & 1u)) >> 11;
  const int f = 1023 + 63 - lz + sh;   // exponent field before a carry
  const uint64_t sign = (uint64_t)t & 0x8000000000000000ULL;
  if (f >= 1 && f <= 2045) return bits_as<double>(sign | (((uint64_t)(f - 1) << 52) + u));
  return scalbn((double)t, sh);
}

// (double)h + (double)l of a float pair, |l| <= ulp(h) / 2: added as integers
// on h's grid of 2^-53, which is exact for every pair that split_d made.
__host__ __device__ __forceinline__ double pair_d(float h, float l) {
  const uint32_t hb = bits_as<uint32_t>(h), a = hb & 0x7fffffffu, E = a >> 23;
  if (E - 64u < 190u) {   // h normal, 2^-63 .. 2^126
    const float sl = l * bits_as<float>((307u - E) << 23);   // l / 2^(e - 53), exactly
#ifdef __CUDA_ARCH__
    const int32_t d = __float2int_rn(sl);
#else
    const int32_t d = fabsf(sl) < 1e9f ? (int32_t)lrintf(sl) : 0x7fffffff;
#endif
    const int64_t m = ((int64_t)((a & 0x7fffffu) | 0x800000u) << 30) +
                      ((int32_t)hb < 0 ? -(int64_t)d : (int64_t)d);
    const uint32_t up = (uint32_t)(m >> 53);   // h's own binade: 2^-52, else 2^-53
    if ((float)d == sl && (uint32_t)(d + (1 << 29)) <= (1u << 30) && (up & (uint32_t)m) == 0)
      return bits_as<double>((((uint64_t)(hb & 0x80000000u)) << 32) |
                             (((uint64_t)(E + 894u + up) << 52) + (uint64_t)(m >> up)));
  }
  return f2d(h) + f2d(l);
}

// h = bf16(x) and l = bf16(x - (double)h): the remainder below h is an integer
// of at most 46 bits on x's last place.
__host__ __device__ __forceinline__ void split_bf(double x, __nv_bfloat16 &h, __nv_bfloat16 &l) {
  const uint64_t b = bits_as<uint64_t>(x);
  const uint32_t ex = (uint32_t)(b >> 52) & 0x7ffu, s = (uint32_t)(b >> 48) & 0x8000u;
  if (ex - 950u >= 200u) {   // zero, and where h or l could leave the normal range
    h = d2bf16(x);
    l = d2bf16(x - f2d(__bfloat162float(h)));
    return;
  }
  const uint64_t m = (b & 0xfffffffffffffULL) | (1ULL << 52);
  const uint32_t q = (uint32_t)(m >> 45);
  const uint64_t rem = m & ((1ULL << 45) - 1);
  const uint32_t up = (uint32_t)((rem + (1ULL << 44) - 1 + (q & 1u)) >> 45);
  h = bits_as<__nv_bfloat16>((uint16_t)(s | (((ex - 897u) << 7) + q + up)));
  const int64_t r = (int64_t)rem - (int64_t)((uint64_t)up << 45);
  if (r == 0) {
    l = bits_as<__nv_bfloat16>((uint16_t)0);
    return;
  }
  uint64_t u = (uint64_t)(r < 0 ? -r : r);
  const int lz = clz64(u);
  u <<= lz;
  const uint32_t w = (uint32_t)(u >> 32), t = w >> 24;
  const uint32_t below = (w & 0xffffffu) | ((uint32_t)u != 0 ? 1u : 0u);
  const uint32_t c = (below + 0x7fffffu + (t & 1u)) >> 24;
  const uint32_t sl = s ^ (r < 0 ? 0x8000u : 0u);
  l = bits_as<__nv_bfloat16>((uint16_t)(sl | (((ex - 886u - (uint32_t)lz) << 7) + t + c)));
}

}  // namespace lgw
