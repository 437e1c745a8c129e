"""Raised function attributes are remembered per device and kernel, for any number of threads: the bookkeeping
(csrc/dm_grants.h, host code) compiled and run here, with two devices that forget nothing and grant nothing twice; and no
launcher keeps a flag of its own for the whole process."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_06864_gb300", "csrc")

PROGRAM = r"""
#include "dm_grants.h"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  dm::Grants g;
  int k1, k2, calls = 0;
  auto yes = [&] { ++calls; return true; };
  auto no = [&] { ++calls; return false; };
  g.ensure(0, &k1, 100, yes);
  g.ensure(0, &k1, 100, yes);
  g.ensure(0, &k1, 60, yes);
  if (calls != 1) return 1;
  g.ensure(1, &k1, 100, yes);  // the other device has its own limit
  if (calls != 2) return 2;
  g.ensure(0, &k2, 100, yes);
  g.ensure(0, &k1, 200, yes);
  if (calls != 4) return 3;
  g.ensure(1, &k2, 100, no);  // a failure is no grant
  g.ensure(1, &k2, 100, yes);
  if (calls != 6) return 4;
  std::atomic<int> n{0};
  std::vector<std::thread> t;
  int keys[64];
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&] { for (int r = 0; r < 100; ++r) for (int j = 0; j < 64; ++j) g.ensure(j & 1, keys + j, 8, [&] { ++n; return true; }); });
  for (auto& x : t) x.join();
  return n == 64 ? 0 : 5;
}
"""


def test_per_device_and_kernel(tmp_path):
    src, exe = tmp_path / "grants.cpp", tmp_path / "grants"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_launchers_share_it():
    for name in os.listdir(CSRC):
        if name.endswith(".cu"):
            text = open(os.path.join(CSRC, name)).read()
            assert not re.search(r"static bool \w+ = false", text), name
            assert "cudaFuncAttributeMaxDynamicSharedMemorySize" not in text, name
