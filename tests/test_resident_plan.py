"""Host side of the resident solver's plan (csrc/cgr_plan.h), compiled with the host
compiler: no GPU and no CUDA needed."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_02558_gb300", "csrc")

# a grow-only buffer like the library's device buffer; ensure() throws while `full`
PRELUDE = r"""
#include <cstdio>
#include <cstdlib>
#include "cgr_plan.h"
struct Fake {
  void* p = nullptr;
  size_t cap = 0;
  bool full = false;
  void* ensure(size_t bytes) {
    if (bytes <= cap && p) return p;
    std::free(p);
    p = nullptr;
    cap = 0;
    if (full) throw 1;
    p = std::malloc(bytes);
    cap = bytes;
    return p;
  }
};
"""


def run(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(PRELUDE + "int main() {\n" + body + "\n}\n")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_plan_is_disowned_when_its_buffer_cannot_grow(tmp_path):
    out = run(tmp_path, r"""
  qp::ResidentPlan c;
  Fake b;
  c.room(b, 1000, 128);
  c.chunk = 128;                     // both plan kernels are enqueued
  c.room(b, 900, 128);               // the next solve, in the same room
  std::printf("%d ", c.chunk);
  b.full = true;                     // another precision's plan needs more, and there is none
  try { c.room(b, 2000, 32); std::printf("no-throw "); } catch (int) {}
  b.full = false;
  c.room(b, 1000, 128);              // new memory: nothing in it
  std::printf("%d ", c.chunk);
  c.chunk = 128;
  b.full = true;                     // the same plan after the buffer was lost
  std::free(b.p); b.p = nullptr; b.cap = 0;
  try { c.room(b, 1000, 128); std::printf("no-throw "); } catch (int) {}
  std::printf("%d ", c.chunk);
  b.full = false;
  c.room(b, 1000, 128);
  c.chunk = 128;
  c.room(b, 1001, 128);              // grown: the contents are gone
  std::printf("%d\n", c.chunk);
  std::free(b.p);
""")
    assert out == ["128", "0", "0", "0"]
