"""The occupancy trie's numbering of a slot's children (vg_trie.h), on the CPU: the word and the
bit of every child are slot * 2^7 + child, in 64 bits, up to the largest slot that a call of the
most points a call takes can have (beyond 2^25 slots that product does not fit 32 bits)."""
import os
import shutil
import subprocess

import pytest

from paper_2102_11084_gb300 import build as vgbuild

PROGRAM = r"""
#include <cstdio>
#include "vg_trie.h"
int main() {
  const uint64_t last = uint64_t(vg::trie_slots(vg::kMaxPoints)) - 1;
  const uint64_t slots[] = {0, 1, (1u << 25) - 1, 1u << 25, (1u << 25) + 1, 1u << 27, last};
  for (uint64_t s : slots)
    for (uint32_t d = 0; d <= vg::kTrDigit; ++d)
      if (uint64_t(vg::trie_word(uint32_t(s), d)) * 32 + (d & 31) != (s << vg::kTrDigitBits) + d) {
        std::printf("slot %llu child %u\n", (unsigned long long)s, d);
        return 1;
      }
  return last > (1u << 25) ? 0 : 2;
}
"""


def test_words_of_a_slots_children(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "words.cpp"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(vgbuild._nvcc()))), "include")
    exe = str(tmp_path / "words")
    r = subprocess.run([cxx, "-std=c++17", "-I" + vgbuild.CSRC, "-I" + cuda, str(src), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
