"""Buffers from a caller's allocator of any alignment: on a 16-byte boundary, inside the block the allocator gave, and
that block is what is kept for release; null stays null."""
import subprocess

from paper_1608_03722_gb300 import _build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "alloc.h"
struct Log { size_t off, live, asked; int fail; };
static void* take(size_t n, void* u) {
  Log* l = (Log*)u;
  if (l->fail-- == 0) return nullptr;
  l->asked = n;
  ++l->live;
  return (char*)aligned_alloc(256, (n + 512) & ~(size_t)255) + l->off;
}
static void give(void* p, void* u) { Log* l = (Log*)u; --l->live; free((char*)p - l->off); }
int main() {
  int bad = 0;
  for (size_t off = 0; off < 64; ++off)
    for (int fail = -1; fail < 2; ++fail) {
      Log l = {off, 0, 0, fail};
      dsdna_allocator a = {take, give, &l};
      void* raw = nullptr;
      char* p = (char*)dsdna::alloc16(a, 1024, &raw);
      if (!p) { bad += raw != nullptr || l.live != 0 || fail < 0; continue; }
      bad += (uintptr_t)p % 16 != 0 || p < (char*)raw || p + 1024 > (char*)raw + l.asked || l.live != 1;
      bad += off % 16 == 0 && (p != raw || l.asked != 1024);
      give(raw, &l);
    }
  printf("%d\n", bad);
  return bad != 0;
}
"""


def test_blocks_of_any_alignment(tmp_path):
    (tmp_path / "a.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-I", _build.CSRC, str(tmp_path / "a.cpp"), "-o", str(tmp_path / "a")])
    r = subprocess.run([str(tmp_path / "a")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
