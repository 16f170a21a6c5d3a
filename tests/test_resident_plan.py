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


def test_room_of_a_block(tmp_path):
    """Lists fit the shared memory at every size, hold every contact set up to 512 contacts a
    block, and with all the room the walled boxes that the plan's counts were taken from."""
    out = run(tmp_path, r"""
  const size_t room = 232448 - 4400 - 256;  // a block's most on sm_103a, less the static part
  for (int all = 0; all < 2; ++all)
    for (int chunk = 1; chunk <= qp::CR_CHUNK2; ++chunk) {
      const qp::ResidentShape s = qp::resident_shape(chunk, room, all);
      if (s.smem() > room || s.rcap % 2 || s.nbcap < 1) std::printf("bad-%d-%d ", all, chunk);
      if (chunk <= qp::CR_CHUNK1 && (s.nbcap != 2 * chunk || s.rcap < 2 * chunk || !s.full)) std::printf("short-%d ", chunk);
      if (chunk > qp::CR_CHUNK1 && !s.own_rb && s.rcap * qp::CR_WL > chunk * qp::CR_WR) std::printf("alias-%d ", chunk);
      if (all && !s.full) std::printf("full-%d ", chunk);
    }
  // contacts and bodies a block of walled boxes of 52, 55, 58 and 60 spheres a side
  const int need[4][2] = {{805, 810}, {944, 935}, {1101, 1074}, {1214, 1179}};
  for (auto& n : need) std::printf("%d", qp::resident_shape(n[0], room, true).nbcap >= n[1]);
  // no room at all
  std::printf(" %d\n", qp::resident_shape(1280, 1000, true).nbcap);
""")
    assert out == ["1111", "0"]


def test_refusals_are_remembered_for_the_contact_set(tmp_path):
    out = run(tmp_path, r"""
  using P = qp::ResidentPlan;
  P c;
  c.chunk = 900;
  c.refused(true, false);   // the usual room was too small: all of it next, with another plan
  std::printf("%d%d%d ", c.chunk, c.tried[0] == P::USUAL, c.tried[1] == P::ALL);
  c.chunk = 900;
  c.refused(true, true);    // and so was all of it
  std::printf("%d%d%d ", c.chunk, c.tried[0] == P::USUAL, c.tried[1] == P::NONE);
  c.assembled();
  std::printf("%d%d\n", c.tried[0] == P::USUAL, c.tried[1] == P::ALL);
""")
    assert out == ["011", "011", "11"]
