"""What belongs to a CUDA device (kernel attributes, occupancy) is kept per
device and made once per device, by whichever thread comes first."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1110_1379_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <stdexcept>
#include <thread>
#include <vector>
#include "frmg_perdevice.h"
int main() {
  frmg::PerDevice<int> v;
  std::atomic<int> made[4] = {}, wrong{0};
  try {
    v.get(3, []() -> int { throw std::runtime_error("refused"); });
    return 1;
  } catch (std::runtime_error &) {
  }
  std::vector<std::thread> t;
  for (int q = 0; q < 8; q++)
    t.emplace_back([&]() {
      for (int n = 0; n < 1000; n++) {
        const int d = n % 4;
        if (v.get(d, [&]() { made[d]++; return 10 + d; }) != 10 + d) wrong++;
      }
    });
  for (auto &x : t) x.join();
  for (auto &m : made)
    if (m != 1) return 2;
  return wrong ? 3 : 0;
}
"""


def test_made_once_per_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_process_wide_device_state():
    """Function-local statics that hold what is true of one device only."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as fh:
            for n, line in enumerate(fh, 1):
                if re.match(r"\s+static (thread_local )?(bool|int|long long|unsigned|size_t)\s+\w+\s*(=|;)",
                            line):
                    found.append(f"{os.path.basename(path)}:{n}: {line.strip()}")
    assert not found, found
