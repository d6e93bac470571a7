"""Call numbers of the single-launch force call: whichever grids the calls have, each finds the agreement word it counts
on cleared, and no number comes twice between two clears of the device words."""
import os
import subprocess

from paper_1608_03722_gb300 import _build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "once_calls.h"
using namespace dsdna;
int main(int argc, char** argv) {
  OnceCalls c;
  c.next = argv[1][0] == '-' ? ONCE_CALLS - (unsigned)atoi(argv[1] + 1) : (unsigned)atoi(argv[1]);
  printf("%u\n", c.next);
  for (int k = 0; k < 12; ++k) {
    bool clear = false;
    const unsigned call = c.take(argc > 2 && k == atoi(argv[2]), &clear);
    printf("%u %d\n", call, (int)clear);
  }
}
"""


def _sequence(tmp_path, *args):
    exe = tmp_path / "calls"
    if not exe.exists():
        (tmp_path / "calls.cpp").write_text(SRC)
        subprocess.check_call(["g++", "-std=c++17", "-I", _build.CSRC, str(tmp_path / "calls.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe), *args], capture_output=True, text=True, check=True).stdout.split("\n")
    return int(out[0]), [tuple(map(int, l.split())) for l in out[1:] if l]


def _sound(first, calls, grids, tags=True):
    """The kernel's agreement (res_publish, res_agree): call c counts its blocks on word (c + 1) mod 3 and clears the word
    before it; its records carry the low 30 bits of c + 1.  True when every call starts its count from zero and, between
    clears, no tag comes twice (nor that of cleared records, zero)."""
    words, seen = [0, 0, 0], {0}
    words[first % 3] = grids[-1]                     # left by the call before
    for (call, clear), grid in zip(calls, grids):
        if clear:
            words, seen = [0, 0, 0], {0}
        p = (call + 1) % 2 ** 32
        if words[p % 3] != 0 or (tags and p % 2 ** 30 in seen):
            return False
        seen.add(p % 2 ** 30)
        words[p % 3] += grid
        words[(p + 2) % 3] = 0
    return True


GRIDS = [3, 152, 1, 40, 152, 2, 7, 152, 3, 9, 1, 100]


def test_numbers_start_over_cleanly(tmp_path):
    for args in (["0"], ["1"], ["-1"], ["-2"], ["-5"], ["-5", "2"], ["7", "3"], ["-3", "3"], ["0", "0"]):
        first, calls = _sequence(tmp_path, *args)
        assert any(c for _, c in calls) == (args[0][0] == "-" or len(args) > 1)
        assert _sound(first, calls, GRIDS), args


def test_a_bare_32_bit_count_is_not_sound():
    """The model sees what a counter without clears does: 2^32 is no multiple of 3, and tags have 30 bits."""
    assert not _sound(2 ** 32 - 5, [(c % 2 ** 32, 0) for c in range(2 ** 32 - 5, 2 ** 32 + 7)], GRIDS, tags=False)
    assert not _sound(2 ** 30 - 5, [(c, 0) for c in range(2 ** 30 - 5, 2 ** 30 + 7)], GRIDS)
    assert _sound(100, [(c, 0) for c in range(100, 112)], GRIDS)
