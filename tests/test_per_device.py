"""CPU check of what the library keeps for each GPU of a process, with devices that only exist in
the test: a second device is set up on its own, a failure is not remembered, threads set up once."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_02060_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
#define CHECK(c) if (!(c)) return std::printf("line %d: %s\n", __LINE__, #c), 1
int main() {
  lddmm::PerDevice<bool> set;
  int made[70] = {};
  bool fail = true;
  auto use = [&](int dev) { return set.get(dev, [&] { ++made[dev < 0 ? 69 : dev]; return !fail; }); };
  CHECK(!use(0) && !use(0) && made[0] == 2);          // a failure is tried again
  fail = false;
  CHECK(use(0) && use(0) && made[0] == 3);            // and a success kept
  CHECK(made[1] == 0 && use(1) && made[1] == 1);      // the second device is set up too
  CHECK(use(63) && use(63) && made[63] == 1);
  CHECK(use(64) && use(64) && made[64] == 2);         // past the kept ones: every time
  CHECK(use(-1) && use(-1) && made[69] == 2);
  lddmm::PerDevice<int> num;
  CHECK(num.get(0, [] { return 152; }) == 152 && num.get(1, [] { return 7; }) == 7);
  CHECK(num.get(0, [] { return 9; }) == 152);
  lddmm::PerDevice<int> shared;
  std::atomic<int> calls{0}, wrong{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 1000; ++i)
        if (shared.get(t & 1, [&] { ++calls; return 10 + (t & 1); }) != 10 + (t & 1)) ++wrong;
    });
  for (auto& t : ts) t.join();
  CHECK(calls == 2 && wrong == 0);
  return 0;
}
"""


def test_values_are_kept_for_each_device(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "kept.cpp", tmp_path / "kept"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-O1", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_device_calls_go_through_what_is_kept_for_each_device():
    """A kernel's limit and the SM count are asked for in one place, beside PerDevice."""
    for call in ("cudaFuncSetAttribute(", "cudaDeviceGetAttribute("):
        found = {os.path.basename(path): n for path in glob.glob(os.path.join(CSRC, "*"))
                 if (n := re.sub(r"//[^\n]*", "", open(path).read()).count(call))}
        assert found == {"kernels.h": 1}, (call, found)
