"""Kernel set-up that holds for one device (function attributes, occupancy) is
found once for each, from any number of threads, and every launcher that sets an
attribute keeps it so."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_07508_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  static sao::PerDevice<int> known;
  std::atomic<int> asked[66] = {};
  std::atomic<int> wrong{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 8; ++t)
    threads.emplace_back([&] {
      for (int round = 0; round < 100; ++round)
        for (int d = 0; d < 64; ++d)
          if (known.get(d, [&] { asked[d]++; return 1000 + d; }) != 1000 + d) wrong++;
    });
  for (auto &t : threads) t.join();
  for (int d = 0; d < 64; ++d)
    if (asked[d] != 1) wrong++;
  for (int i = 0; i < 3; ++i)
    if (known.get(65, [&] { return asked[65]++; }) != i) wrong++;
  std::printf("%d\n", wrong.load());
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_found_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"


def test_attributes_are_set_on_every_device():
    sites = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"cudaFuncSetAttribute\(", code):
            sites += 1
            before = code[max(0, m.start() - 500):m.start()]
            assert re.search(r"PerDevice<|once_flag once\[\d+\]\[kMaxDevices\]", before), f"{name}: set once per process"
    assert sites >= 3
