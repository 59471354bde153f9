"""The integer-pipe conversions of csrc/fp_bits.cuh against the native ones, bit for bit:
random bit patterns, ties and near ties, exponents around every fast-path limit, zeros,
subnormals, infinities.  Host code of the same header (no GPU)."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "fp_bits.cuh"
using namespace lgw;
static long bad = 0;
static void both(double x) {
  if (std::isnan(x)) return;
  float h, l;
  split_d(x, h, l);
  const float h0 = (float)x, l0 = (float)(x - (double)h0);
  if (bits_as<uint16_t>(d2bf16(x)) != bits_as<uint16_t>(__double2bfloat16(x)) && bad++ < 10)
    printf("bf16 %a\n", x);
  const bool lo = std::isinf(h0) || bits_as<uint32_t>(l) == bits_as<uint32_t>(l0);
  if (bits_as<uint32_t>(d2f(x)) != bits_as<uint32_t>(h0) ||
      bits_as<uint32_t>(h) != bits_as<uint32_t>(h0) || !lo) {
    if (bad++ < 10) printf("%a: %a %a against %a %a\n", x, h, l, h0, l0);
  }
}
// bf16(x) and bf16 of the rest; an integer scaled by a power of two
static void more(double x, uint64_t u) {
  if (std::isnan(x) || std::isinf(x)) return;
  __nv_bfloat16 h, l;
  split_bf(x, h, l);
  const __nv_bfloat16 h0 = __double2bfloat16(x);
  const bool inf = std::isinf(__bfloat162float(h0));
  const __nv_bfloat16 l0 = __double2bfloat16(x - (double)__bfloat162float(h0));
  if ((bits_as<uint16_t>(h) != bits_as<uint16_t>(h0) ||
       (!inf && bits_as<uint16_t>(l) != bits_as<uint16_t>(l0))) && bad++ < 10)
    printf("split_bf %a\n", x);
  const long long t = (long long)u >> (u & 63);
  const int sh = (int)(u >> 8 & 1023) - 512;
  if (bits_as<uint64_t>(ll2d_scaled(t, sh)) != bits_as<uint64_t>(std::scalbn((double)t, sh)) &&
      bad++ < 10)
    printf("ll2d %lld %d\n", t, sh);
}
static void pair(float h, float l) {
  if (std::isnan(h) || std::isnan(l) || std::isnan(h + l)) return;
  if (bits_as<uint64_t>(pair_d(h, l)) != bits_as<uint64_t>((double)h + (double)l) && bad++ < 10)
    printf("pair %a %a\n", h, l);
}
static void wide(float x) {
  if (!std::isnan(x) && bits_as<uint64_t>(f2d(x)) != bits_as<uint64_t>((double)x) && bad++ < 10)
    printf("f2d %a\n", x);
}
int main() {
  std::mt19937_64 g(1);
  for (long i = 0; i < 2000000; ++i) {
    const uint64_t u = g();
    both(bits_as<double>(u));
    wide(bits_as<float>((uint32_t)u));
    const uint64_t v = (g() & 0x800fffffffffffffULL) | ((850 + u % 400) << 52);
    const uint64_t t = (v & ~0x1fffffffULL) | 0x10000000ULL;      // halfway between floats
    const uint64_t m = (v & ~0x1fffffffffffULL) | 0x100000000000ULL;   // halfway between bf16
    both(bits_as<double>(m)), both(bits_as<double>(m + 1)), both(bits_as<double>(m - 1));
    const uint64_t near[] = {v, t, t + 1, t - 1, v | 0x000ffffff0000000ULL, v & ~0x1fffffffULL};
    for (uint64_t w : near) {
      const double x = bits_as<double>(w);
      float h, l;
      both(x), more(x, g());
      split_d(x, h, l);
      pair(h, l), pair(h, -l), pair(h, std::ldexp(l, (int)(u & 7) - 3));
    }
    more(bits_as<double>(u), u);
    const uint64_t rest[] = {m, m + 1, m - 1, m + 0x8000000000ULL, m & ~0xfffffffffULL};
    for (uint64_t w : rest)
      more(bits_as<double>(w), w);
    pair(bits_as<float>((uint32_t)u), bits_as<float>((uint32_t)(u >> 32)));
  }
  const double ms[] = {1.0, 0x1.fffffep0, 0x1.fffffefp0, 0x1.ffffffp0, 0x1.0000008p0};
  for (int e = -1074; e <= 1023; ++e)
    for (double m : ms) {
      const double x = std::ldexp(m, e);
      both(x), both(-x), wide((float)x), wide((float)-x);
      more(x, 1ULL << (e & 63)), more(-x, 3);
      const float f = (float)x;
      pair(f, std::ldexp(f, -24)), pair(f, -std::ldexp(f, -24)), pair(f, -std::ldexp(f, -25)), pair(-f, f * 0x1p-40f);
    }
  const double sp[] = {0.0, -0.0, INFINITY, -INFINITY};
  for (double x : sp) both(x), wide((float)x), pair((float)x, 0.0f);
  printf("bad %ld\n", bad);
  return bad != 0;
}
"""


def test_conversions_match_the_native_ones():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cu"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(PROGRAM)
        inc = os.path.join(ROOT, "paper_2310_20103_gb300", "csrc")
        subprocess.run([nvcc, "-O2", "-std=c++17", "-I" + inc, "-o", exe, src], check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout
