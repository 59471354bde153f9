// Digits of FP64 values for the tensor-core products (k_gemm_oz.cu).
#pragma once

#include "lgw_internal.cuh"

namespace lgw {
namespace oz {

constexpr int S = OZ_SLICES;

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x on the grid 2^(f - 1022 - 55) of a row whose largest exponent field is f,
// biased so that the base-128 digits come out as 64 + d_s.
__device__ __forceinline__ unsigned long long fixed56(double x, int f) {
  constexpr unsigned long long bias =
      64ULL * ((1ULL << 49) + (1ULL << 42) + (1ULL << 35) + (1ULL << 28) + (1ULL << 21) +
               (1ULL << 14) + (1ULL << 7) + 1ULL);
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffLL;
  if (ex != 0) m |= 1LL << 52;
  const int sh = max(ex, 1) - f + 2;   // at most 2: |x| < 2^(f - 1022), or x is 0
  long long v = 0;
  if (sh >= 0)
    v = m << min(sh, 2);
  else if (sh > -56)
    v = (m + (1LL << (-sh - 1))) >> -sh;
  if (b < 0) v = -v;
  return (unsigned long long)v + bias;
}
// BF16 bits of 2^(-7s) times digit s (an integer in [-64, 64]) of the biased
// fixed point
__device__ __forceinline__ uint32_t digit_bf16(unsigned long long u, int s) {
  const uint32_t t = s == 0 ? (uint32_t)(u >> 49) : (uint32_t)(u >> (49 - 7 * s)) & 127u;
  const float w = __uint_as_float((uint32_t)(127 - 7 * s) << 23);   // 2^(-7s)
  return __float_as_uint((__uint_as_float(0x4B000000u | t) - 8388672.0f) * w) >> 16;
}

// Two adjacent K elements e, e + 1 (e even) of operand row `row`, whose
// largest exponent field is f.
__device__ __forceinline__ void store_digits2(double x, double y, int f, int row, int e,
                                              const OzOperand &o) {
  const unsigned long long u0 = fixed56(x, f), u1 = fixed56(y, f);
  const size_t plane = (size_t)o.nkb * o.rows * 64;
  uint16_t *dst = o.d + ((size_t)(e >> 6) * o.rows + row) * 64 + (e & 63);
#pragma unroll
  for (int s = 0; s < S; ++s)
    *reinterpret_cast<uint32_t *>(dst + s * plane) =
        digit_bf16(u0, s) | (digit_bf16(u1, s) << 16);
}

}  // namespace oz
}  // namespace lgw
