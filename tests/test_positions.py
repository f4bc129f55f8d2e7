"""The kernels' arithmetic on key positions (csrc/kvd_positions.h), against 64-bit arithmetic over the ends of the int range,
compiled for the host with signed overflow trapped.

A segment may end at the largest int and a query may stand there ("sees every key"): a sum of a block's position and its
length overflows in the last block, and an absent segment then looked as if it held the block."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_19664_b200", "csrc")

PROGRAM = r"""
#include <climits>
#include <cstdint>
#include <initializer_list>
#include "kvd_positions.h"
using namespace kvd;
int main() {
  const int at[] = {INT_MIN, INT_MIN + 1, -1, 0, 1, 63, 64, 65, 100, 127, 128, 1 << 20, INT_MAX - 129, INT_MAX - 128, INT_MAX - 127,
                    INT_MAX - 64, INT_MAX - 63, INT_MAX - 62, INT_MAX - 1, INT_MAX};
  const int blocks[] = {0, 64, 128, 1 << 20, INT_MAX - 127, INT_MAX - 63};
  const int lens[] = {0, 1, 63, 64, 65, 128, 1000, INT_MAX - 64, INT_MAX};
  for (int qp : at)
    for (int window : lens) {
      const int64_t first = window > 0 ? static_cast<int64_t>(qp) - window + 1 : 0;
      if (first_visible(qp, window) != (first > 0 ? first : 0)) return 1;
    }
  for (int pos0 : blocks) {
    for (int first : at)
      for (int len : lens) {
        if (first < 0 || static_cast<int64_t>(first) + len > INT_MAX) continue;
        unsigned long long bits = 0;
        for (int k = 0; k < 64; ++k)
          if (first <= static_cast<int64_t>(pos0) + k && static_cast<int64_t>(pos0) + k < static_cast<int64_t>(first) + len) bits |= 1ull << k;
        if (segment_slots(first, len, pos0) != bits) return 2;
        for (int n : {1, 32, 64, 128})
          if (segment_holds(first, len, pos0, n) != (first <= pos0 && static_cast<int64_t>(pos0) + n <= static_cast<int64_t>(first) + len)) return 3;
      }
    for (int last : at)
      for (int n : {1, 32, 64, 128})
        if (ends_by(pos0, n, last) != (static_cast<int64_t>(pos0) + n - 1 <= last)) return 5;
    for (int lo : at)
      for (int qp : at) {
        if (lo < 0) continue;
        unsigned long long bits = 0;
        for (int k = 0; k < 64; ++k)
          if (lo <= static_cast<int64_t>(pos0) + k && static_cast<int64_t>(pos0) + k <= qp) bits |= 1ull << k;
        if (visible_slots(lo, qp, pos0) != bits) return 4;
      }
  }
  return 0;
}
"""


def test_positions_over_the_whole_int_range(tmp_path):
    src, exe = tmp_path / "positions.cpp", tmp_path / "positions"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error", "-I", CSRC, "-o",
                    str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.parametrize("name", ["kvd_attention.cu", "kvd_prefill_attention.cu", "kvd_prefill_attention_tc.cu", "kvd_api.cu"])
def test_kernels_add_no_length_to_a_position_they_compare(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    sums = re.findall(r"(?:pos0|pos_first) \+ \w+ <=? |(?:pos0|pos_first) \+ \w+ >=? ", text)
    assert not sums  # (pos0 + PT_KEYS - 1, a block's last position, is in range)
    assert not re.search(r"- [\w.>-]*window \+ 1", text)
