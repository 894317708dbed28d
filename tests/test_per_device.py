"""Per-device set-up (csrc/qlin_per_device.h): each device's value is made once, by
the first call on that device, also when threads race for it.  Compiled and run
on the CPU; kernel attributes and occupancy are kept in it."""
import os
import re
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2609_21849_gb300", "csrc")
MAIN = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "qlin_per_device.h"
std::atomic<int> made[qlin::kMaxDevices];
int value(int dev) {
  static qlin::PerDevice<int> v;   // as the launchers keep theirs
  return v.get(dev, [&] { ++made[dev]; return 100 + dev; });
}
int main() {
  std::atomic<int> bad{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 2 * qlin::kMaxDevices; ++i) {
        const int dev = (i + 7 * t) % qlin::kMaxDevices;
        if (value(dev) != 100 + dev) ++bad;
      }
    });
  for (auto& t : ts) t.join();
  for (int d = 0; d < qlin::kMaxDevices; ++d) bad += made[d] != 1;
  std::printf("%d\n", bad.load());
}
"""


def test_one_value_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I" + CSRC, str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.strip() == "0"


@pytest.mark.parametrize("name", ["qlin_gemm.cu", "qlin_quant.cu"])
def test_no_attribute_is_set_once_per_process(name):
    # a static initialised by cudaFuncSetAttribute or an occupancy query would
    # hold the first device's answer for all
    src = open(os.path.join(CSRC, name)).read()
    assert "PerDevice<" in src and "cudaFuncSetAttribute" in src
    assert not re.search(r"static[^;{}]*=\s*cuda(FuncSetAttribute|Occupancy)", src)
    assert "std::call_once(once, [&]" not in src
