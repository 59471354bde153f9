"""Split counts and partial buffers of the sliced FP64 products (csrc/oz_plan.cuh), on the CPU.

A contraction of more than 1024 vectors runs in slices of 1024 and a shorter last one, each
with the split count of its own width.  Every slice must fit the buffer that was planned for
all of them: fewer columns get more splits, and often more partial rows in total."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "oz_plan.cuh"
using namespace lgw::oz;
int main() {
  const int SLICE = 1024;
  long bad = 0, first_only = 0;
  for (int nsm : {132, 148, 152})
    for (int nvc = 128; nvc <= 131072; nvc = nvc < 4096 ? nvc + 128 : nvc * 2)
      for (int A = 128; A <= 2048; A += 128)
        for (int rows = 16; rows <= 4112; rows += 16) {
          const int nkb = nvc / KB;
          const size_t have = part_rows(A, rows, SLICE, nkb, nsm);
          const int w = std::min(rows, SLICE);
          const size_t first = (size_t)k_splits(A, w, nkb, nsm) * w;
          bool over = false;
          for (int r0 = 0; r0 < rows; r0 += SLICE) {
            const int nr = std::min(SLICE, rows - r0);
            const size_t need = (size_t)k_splits(A, nr, nkb, nsm) * nr;
            if (need > have && bad++ < 5)
              printf("N %d A %d rows %d slice %d: %zu rows of %zu\n", nvc, A, rows, nr, need, have);
            over = over || need > first;
          }
          first_only += over;
        }
  printf("%ld %ld\n", bad, first_only);
  // widths whose last slice needs several times the first one's rows
  const int c[][3] = {{4096, 384, 1920}, {32768, 896, 4032}, {4096, 1024, 1344}, {2048, 2048, 1424}};
  for (auto &x : c)
    printf("%zu %zu\n", (size_t)k_splits(x[1], SLICE, x[0] / KB, 152) * SLICE,
           part_rows(x[1], x[2], SLICE, x[0] / KB, 152));
  return bad != 0;
}
"""


def test_every_slice_fits_the_planned_partials():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(PROGRAM)
        inc = os.path.join(ROOT, "paper_2310_20103_gb300", "csrc")
        subprocess.run([cxx, "-O2", "-std=c++17", "-I" + inc, "-o", exe, src], check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    lines = r.stdout.split("\n")
    assert int(lines[0].split()[1]) > 0       # the first slice alone would not have been enough
    for ln in lines[1:5]:
        first, planned = map(int, ln.split())
        assert planned > first, r.stdout
