"""State kept per device (csrc/per_device.cuh), on the CPU: a kernel attribute is set on every
device that launches the kernel, also when threads come together, and none launches before."""
import os
import re
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_20103_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
using namespace lgw;
int main() {
  static DeviceOnce once;
  static DeviceValue value;
  static std::atomic<int> set[70];
  std::atomic<int> bad{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 2000; ++i) {
        const int dev = (i * 7 + t) % 70;
        once(dev, [&] { set[dev]++; });
        if (set[dev] == 0) bad++;                       // returned before it was set
        if (value(dev, [&] { return 100 + dev; }) != 100 + dev) bad++;
      }
    });
  for (auto &t : ts) t.join();
  for (int d = 0; d < 64; ++d)
    if (set[d] < 1 || set[d] > 8) bad++;                // once, or where threads met
  once(3, [&] { bad++; });
  printf("%d\n", bad.load());
  return bad != 0;
}
"""


def test_every_device_is_set_before_its_first_use():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(PROGRAM)
        subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I" + CSRC, "-o", exe, src],
                       check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_kept_per_process():
    """Kernel attributes are set through DeviceOnce only, never behind a flag of the process."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert not re.search(r"static (bool|int) \w+ = (false|0);", text), name
