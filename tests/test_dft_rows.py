"""CPU check of where a table's rows lie, on axes whose tables hold more than 2^31 elements."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_02060_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "dft_rows.cuh"
int main(int argc, char** argv) {
  for (int i = 1; i + 1 < argc; i += 2)
    std::printf("%llu\n", lddmm::fold_row_bytes(std::atoi(argv[i]), 4u * (unsigned)std::atoi(argv[i + 1])));
}
"""


def test_entries_of_long_axes(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    # the longest axis a grid can have: 3 n ny nz < 2^31 with ny = nz = 2
    cases = [(p, n) for n in (2, 3, 8, 264, 46340, 46341, 50001, 200000, 178956970) for p in (0, 1, n // 2)]
    r = subprocess.run([str(exe)] + [str(k) for c in cases for k in c], capture_output=True, text=True, check=True)
    want = [4 * n * max(2 * p - 1, 0) for p, n in cases]
    assert [int(w) for w in r.stdout.split()] == want and max(want) > 2 ** 33


def test_k_fold_forms_table_offsets_there():
    s = open(os.path.join(CSRC, "kernels_dft.cu")).read()
    assert s.count("col + fold_row_bytes(p, n4)") == 2
    assert s.count("a.R + m)") == s.count("a.R +") == 2
