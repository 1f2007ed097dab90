"""CPU check of the range test that lets a kernel, not a checked copy, touch a caller's buffer."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_02060_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "memory_span.h"
#define CHECK(c) if (!(c)) return std::printf("line %d: %s\n", __LINE__, #c), 1
int main() {
  using lddmm::span_holds;
  const uint64_t top = ~0ull, b = 0x7f0000000000ull;
  CHECK(span_holds(b, 100, b, 100) && span_holds(b, 100, b + 40, 60) && span_holds(b, 100, b + 100, 0));
  CHECK(!span_holds(b, 100, b, 101) && !span_holds(b, 100, b + 40, 61) && !span_holds(b, 100, b + 101, 0));
  CHECK(!span_holds(b, 100, b - 1, 50) && !span_holds(b, 0, b, 1));
  CHECK(!span_holds(b, 100, b + 4, top) && !span_holds(b, 100, b + 4, top - 3));   // no wrap around
  CHECK(span_holds(top - 99, 100, top - 49, 50) && !span_holds(top - 99, 100, top - 49, 51));
  return 0;
}
"""


def test_span(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "span.cpp", tmp_path / "span"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_velocity_kernels_touch_whole_spans_only():
    """Both one-pass conversions of a caller's field ask for all of its bytes."""
    s = open(os.path.join(CSRC, "lddmm_api.cu")).read()
    for call, ptr in (("launch_store_checked(src, ctx->v, n,", "src"), ("launch_from_storage(ctx->v, dst, n,", "dst")):
        i = s.index(call)
        guard = s.rindex("if (is_local_", 0, i)
        assert s[guard:].startswith("if (is_local_span(%s, n * sizeof(float)))" % ptr), call
        assert re.search(r"const int64_t n = \(int64_t\)ctx->p\.T \* 3 \* g\.N;", s[s.rindex("\n}", 0, guard):guard])
