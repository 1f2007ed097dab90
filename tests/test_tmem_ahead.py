"""CPU check of the order in which the chunk-ahead TMEM reads name their registers: a model of the
asynchronous load, whose registers hold garbage from the issue until the wait that names them."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_02060_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include "tmem_ahead.cuh"
struct Model {
  static const uint32_t* regs[4];
  static uint32_t addr[4];
  static int in_flight, issued;
  static uint32_t value(uint32_t a, int j) { return a * 1000u + (uint32_t)j; }
  static void issue(uint32_t a, uint32_t (&u)[16]) {
    for (int j = 0; j < 16; ++j) u[j] = 0xdeadbeefu;
    regs[in_flight] = u;
    addr[in_flight++] = a;
    ++issued;
  }
  static void wait(uint32_t (&u)[16]) {
    // every load has finished; what the wait does not name stays undefined in the program
    for (int k = 0; k < in_flight; ++k)
      for (int j = 0; j < 16; ++j)
        if (regs[k] == u) u[j] = value(addr[k], j);
    in_flight = 0;
  }
};
const uint32_t* Model::regs[4];
uint32_t Model::addr[4];
int Model::in_flight = 0, Model::issued = 0;

int main() {
  for (int n = 0; n <= 17; ++n) {
    Model::in_flight = Model::issued = 0;
    lddmm::TmemAhead<Model> tm;
    if (n > 0) tm.first(7u);
    for (int k = 0; k < n; ++k) {
      if (k + 1 < n) tm.ahead(7u + (uint32_t)(k + 1));
      if (Model::issued != (k + 2 < n ? k + 2 : n)) return std::printf("n %d: chunk %d not ahead\n", n, k), 1;
      for (int j = 0; j < 16; ++j)
        if (tm.u[j] != Model::value(7u + (uint32_t)k, j)) return std::printf("n %d chunk %d\n", n, k), 1;
      if (k + 1 < n) tm.advance();
    }
    if (Model::in_flight) return std::printf("n %d: a load is left in flight\n", n), 1;
  }
  return 0;
}
"""


def test_registers_are_read_after_the_wait_that_names_them(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL)
    subprocess.run([cc, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_loads_without_their_wait_go_through_tmem_ahead_only():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        s = re.sub(r"//[^\n]*", "", open(path).read())
        # a load and its wait are one statement, but for the two halves TmemAhead is given
        split_loads = [m for m in re.findall(r"asm volatile\((.*?)\);\n", s, flags=re.S)
                       if "tcgen05.ld." in m and "tcgen05.wait::ld" not in m]
        assert len(split_loads) == (1 if path.endswith("tc_ptx.cuh") else 0), path
        calls = re.findall(r"(?:TmemLd16::\w+|tmem_issue16|tmem_wait16)\s*\(", s)
        assert not calls, (path, calls)
