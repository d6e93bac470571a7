"""Heads of the resident kernel's cell lists: a head is found by the rebuild that wrote it and by no other, and zeroed
heads by none, also 2^32 rebuilds later."""
import subprocess

from paper_1608_03722_gb300 import _build

SRC = r"""
#include <cstdio>
#include "cell_heads.h"
using namespace dsdna;
int main() {
  typedef unsigned long long ull;
  const ull near[] = {1, 2, 3, 1ull << 31, (1ull << 32) - 1, 1ull << 32, (1ull << 32) + 1, (1ull << 32) + 3, 3ull << 32, (1ull << 44) - 1};
  const unsigned ids[] = {0, 1, 4864, 77824 + 4864, (1u << RES_ID_BITS) - 1};
  int bad = 0;
  for (ull e : near) {
    bad += res_first(0ull, e) != RES_NONE;
    for (unsigned id : ids)
      for (ull w : near) bad += res_first(res_head(w, id), e) != (w == e ? id : RES_NONE);
  }
  printf("%d\n", bad);
  return bad != 0;
}
"""


def test_heads_match_their_own_rebuild_only(tmp_path):
    (tmp_path / "heads.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-I", _build.CSRC, str(tmp_path / "heads.cpp"), "-o", str(tmp_path / "heads")])
    r = subprocess.run([str(tmp_path / "heads")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
