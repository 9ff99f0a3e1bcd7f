"""Settings that hold for one device are made on every device of a process.

The opt-in to large shared memory is a setting of the current device; it was
remembered once for the whole process, so a second context on another device
failed at its first launch.  The header that remembers it now has no CUDA in
it and runs here, with the devices as plain numbers.
"""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2407_18947_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  rtcc3::PerDevice done;
  std::vector<int> count(70, 0);
  for (int round = 0; round < 3; ++round)
    for (int dev : {0, 1, 5, 63, 0, 1}) done.once(dev, [&] { ++count[dev]; });
  for (int dev : {0, 1, 5, 63}) if (count[dev] != 1) return 1;
  // beyond the mask: made every time
  for (int k = 0; k < 3; ++k) done.once(69, [&] { ++count[69]; });
  if (count[69] != 3) return 2;
  // one that failed is not remembered
  int tries = 0;
  for (int k = 0; k < 3; ++k)
    try { done.once(7, [&] { if (++tries == 1) throw 1; }); } catch (int) {}
  if (tries != 2) return 3;
  // several threads: at least once for every device before any thread goes on
  rtcc3::PerDevice shared;
  std::atomic<int> set[8] = {}, missing{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] {
      for (int k = 0; k < 800; ++k) {
        shared.once(k % 8, [&] { ++set[k % 8]; });
        if (!set[k % 8]) ++missing;
      }
    });
  for (auto& t : ts) t.join();
  return missing ? 4 : 0;
}
"""


def test_made_once_on_every_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_kernel_remembers_its_setting_for_the_whole_process():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+(bool|std::atomic<bool>)\s+attr", text), name
