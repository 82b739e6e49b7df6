"""Kernel attributes and grid sizes are found once on each device, not once per
process (CPU: the launchers' cache, and that every launcher goes through it)."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_12199_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
static std::atomic<int> calls{0};
static int launcher(int dev) {  // as the launchers: one cache per function
  static mstgpu::PerDevice cache;
  return cache.get(dev, [&] { ++calls; return 100 * dev; });
}
int main() {
  std::vector<std::thread> threads;
  std::atomic<int> wrong{0};
  for (int t = 0; t < 8; ++t)
    threads.emplace_back([&] {
      for (int i = 0; i < 3000; ++i)
        if (launcher(i % 3) != 100 * (i % 3)) ++wrong;
    });
  for (auto &t : threads) t.join();
  std::printf("%d %d", wrong.load(), calls.load());
  launcher(63), launcher(63);                    // the last ordinal that is kept
  std::printf(" %d", calls.load());
  launcher(64), launcher(64), launcher(-1);      // past the table: asked for every time
  std::printf(" %d\n", calls.load());
}
"""


def test_a_value_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    assert [int(x) for x in out] == [0, 3, 4, 7]


def test_every_launcher_sets_attributes_per_device():
    """Each cudaFuncSetAttribute is in a find() that PerDevice::get runs, or in a function such a find() calls."""
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        finds = [text[m.start():text.index("});", m.start())] for m in re.finditer(r"\.get\(current_device\(\),", text)]
        called = {name for f in finds for name in re.findall(r"(\w+)\s*(?:<[^<>;]*>)?\(", f)}
        inside = sum(f.count("cudaFuncSetAttribute(") for f in finds)
        for name in called:
            for m in re.finditer(r"\n(?:static )?int " + name + r"\([^;{]*\) \{", text):
                inside += text[m.start():text.index("\n}", m.start())].count("cudaFuncSetAttribute(")
        total = text.count("cudaFuncSetAttribute(")
        assert inside == total, path
        seen += total
    assert seen >= 7
