"""Pinned result slots: distinct and 64 bytes apart, pages come when all slots are taken and go with their last one, and a
slot can be given back by the program's last static destructor (under the address sanitizer)."""
import subprocess

from paper_1608_03722_gb300 import _build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include "host_slots.h"
static int pages = 0, most = 0, bad = 0;
static void* get() { if (pages == 4) return nullptr; ++pages; most = pages > most ? pages : most; return aligned_alloc(4096, 4096); }
static void put(void* p) { --pages; free(p); }
static dsdna::HostSlots& slots() { return dsdna::host_slots<get, put>(); }
struct Late { double* slot = nullptr; ~Late() { if (slot) slots().give(slot); if (pages || bad) _Exit(3); } };
static Late late;   // constructed before the slots' first use, so destroyed after anything they might destroy
int main() {
  std::set<double*> live;
  for (int k = 0; k < 256; ++k) {
    double* s = slots().take();
    bad += !s || (size_t)s % 64 != 0 || !live.insert(s).second;
    s[7] = k;
  }
  bad += pages != 4 || slots().take() != nullptr;
  int n = 0;
  for (double* s : live) if (++n % 2) slots().give(s);            // every page half empty: none goes
  bad += pages != 4;
  double* extra = slots().take();
  bad += !extra;
  n = 0;
  for (double* s : live) if (++n % 2 == 0) slots().give(s);
  bad += pages != 1;                                              // the one that holds `extra`
  late.slot = slots().take();
  slots().give(extra);
  bad += pages != 1;
  printf("%d %d\n", bad, pages);
  return bad != 0;
}
"""


def test_slots(tmp_path):
    (tmp_path / "s.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-g", "-fsanitize=address", "-I", _build.CSRC, str(tmp_path / "s.cpp"), "-o",
                           str(tmp_path / "s")])
    r = subprocess.run([str(tmp_path / "s")], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
