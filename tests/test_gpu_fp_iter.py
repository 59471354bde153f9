"""The reciprocal, inverse square root, square root and quotient of csrc/fp_iter.cuh against
CUDA's own operations, in units of the last place.

Bounds, from the iterations: the hardware's estimates err by 2^-20 (the PTX manual's bound),
a third-order step leaves 2^-60 and rounds once, so the reciprocal is within one unit of the
rounded quotient; the inverse root rounds d y before its residual, half a unit more on each
side, and CUDA's rsqrt errs by one: three units between them; the corrected square root and
quotient have exact residuals, so within one unit again.  Whole exponent range, values next
to powers of two, the limits of the fast forms, zero and infinity for the reciprocal."""
import os
import shutil
import subprocess
import tempfile

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "fp_iter.cuh"
using namespace lgw;
// distance in representable values; NaN agrees with NaN only
__device__ long long ulps(double a, double b) {
  if (a != a || b != b) return (a != a && b != b) ? 0 : 1LL << 40;
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  const long long u = x < 0 ? (long long)0x8000000000000000ULL - x : x;
  const long long v = y < 0 ? (long long)0x8000000000000000ULL - y : y;
  return u > v ? u - v : v - u;
}
__device__ unsigned long long mix(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__global__ void check(unsigned long long *worst, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long a = mix(2ull * i), b = mix(2ull * i + 1);
  unsigned long long m = a & 0xfffffffffffffULL;
  if ((a >> 60) == 0) m = b & 3;                              // just above a power of two
  if ((a >> 60) == 1) m = 0xffffffffffffcULL | (b & 3);       // just below the next
  // any positive number, subnormals, infinity and NaN
  const double d = __longlong_as_double((long long)((b >> 53) << 52 | m));
  atomicMax(&worst[0], (unsigned long long)ulps(pole_rcp(d), 1.0 / d));
  // 1e-280 .. 1e280
  const int ex = 1023 - 930 + (int)(b % 1860);
  const double x = __longlong_as_double((long long)((unsigned long long)ex << 52 | m));
  if (!(x > 1e-280 && x < 1e280)) return;
  const double r = rsqrt_iter(x), s = sqrt_from(x, r);
  atomicMax(&worst[1], (unsigned long long)ulps(r, rsqrt(x)));
  atomicMax(&worst[2], (unsigned long long)ulps(s, sqrt(x)));
  // a quotient by the root, numerator of any sign within 2^200 of it
  const double num = ldexp((double)(long long)mix(b), (ex - 1023) / 2 - 63 + (int)(a % 400) - 200);
  atomicMax(&worst[3], (unsigned long long)ulps(div_from(num, s, r), num / s));
  // and by a number whose reciprocal is rounded
  const double y = 1.0 / x;
  if (x > 1e-150 && x < 1e150)
    atomicMax(&worst[4], (unsigned long long)ulps(div_from(num, x, y), num / x));
}
int main() {
  unsigned long long *w, h[5] = {};
  const int n = 1 << 26;
  if (cudaMalloc(&w, sizeof h) != cudaSuccess) return 2;
  cudaMemset(w, 0, sizeof h);
  check<<<n / 256, 256>>>(w, n);
  if (cudaMemcpy(h, w, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  printf("%llu %llu %llu %llu %llu\n", h[0], h[1], h[2], h[3], h[4]);
  return 0;
}
"""


def test_iterations_against_the_full_operations():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cu"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(PROGRAM)
        inc = os.path.join(ROOT, "paper_2310_20103_gb300", "csrc")
        subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + inc, "-o", exe, src], check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr)
    rcp, rsq, root, quot, quot2 = map(int, r.stdout.split())
    assert rcp <= 1 and rsq <= 3 and root <= 1 and quot <= 1 and quot2 <= 1, r.stdout
