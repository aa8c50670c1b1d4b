"""The buffer that scoring calls can do without (csrc/fs_optional_buf.h), on the
CPU with an allocator that refuses on demand: a refusal keeps what was there, is
not followed by another request until retry(), and loses nothing."""

import os
import subprocess

from paper_2608_19659_gb300 import _build

HARNESS = r"""
#include <cassert>
#include <cstdlib>
#include "fs_optional_buf.h"
static size_t limit = 100;
static int asked = 0, live = 0;
struct Mem {
  static void* alloc(size_t b) { ++asked; if (b > limit) return nullptr; ++live; return std::malloc(b); }
  static void free(void* p) { --live; std::free(p); }
};
int main() {
  fs::OptionalBuf<Mem> b;
  if (b.ensure(200) || b.p || asked != 1) return 1;         // refused
  if (b.ensure(200) || b.ensure(50) || asked != 1) return 2;  // not asked again, whatever the size
  b.retry();
  if (!b.ensure(50) || b.bytes != 50 || asked != 2) return 3;
  void* p = b.p;
  if (!b.ensure(40) || b.p != p || asked != 2) return 4;    // large enough
  if (b.ensure(150) || b.p != p || b.bytes != 50 || live != 1) return 5;  // a refused growth keeps it
  if (!b.ensure(50) || b.ensure(90) || asked != 3) return 6;
  b.retry();
  if (!b.ensure(90) || b.bytes != 90 || live != 1 || asked != 4) return 7;  // grown: one block
  b.release();
  if (b.p || b.bytes || live) return 8;
  return 0;
}
"""


def test_refusals(tmp_path):
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", _build.CSRC, str(src), "-o", exe], check=True)
    assert os.path.exists(exe)
    r = subprocess.run([exe])
    assert r.returncode == 0, f"step {r.returncode}"
