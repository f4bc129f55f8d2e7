"""The ring of the few-row projection kernel (csrc/kvd_rows_ring.h): stages, and room for two streaming attention CTAs (of the
tensor-core kernel: one, up to 16 rows) beside a CTA that makes keys and values, over all row counts, head sizes and product shapes."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_19664_b200", "csrc")

PROGRAM = r"""
#include "kvd_rows_ring.h"
using namespace kvd;
int main() {
  for (int nr = 8; nr <= RW_MAX_ROWS; nr += 8) {
    const bool many = nr > RW_FEW_ROWS;
    for (int d_head = 64; d_head <= 256; d_head *= 2)
      for (int k_blocks = 1; k_blocks <= 160; ++k_blocks) {
        const int kb = rows_stage_kb(RW_HEAD_TILE, many), steps = (k_blocks + kb - 1) / kb;
        const RowsRing r = rows_ring(nr, RW_HEAD_TILE, kb, d_head, steps);
        const int least = many ? 2 : 3;
        if (r.stages < (steps < least ? steps : least) || r.stages > steps || r.stages > RW_MAX_STAGES) return 1;
        const int attention = d_head == 64 ? 12672 : d_head == 128 ? 16640 : 16512;  // up to four query heads per KV head
        if (r.smem + 1024 + 2 * (attention + 1024) > 228 * 1024) return 2;
        // the tensor-core streaming kernel's CTAs (heads of 64 and 128): four warps' rings of up to four pieces
        if (!many && d_head <= 128 && r.smem + 1024 + 4 * 4 * 4096 + 1024 > 228 * 1024) return 5;
      }
    for (int tile = RW_MIN_TILE; tile <= 256; tile += 8)
      for (int total = 1; total <= 400; total += 7) {
        const int kb = rows_stage_kb(tile, many);
        const RowsRing r = rows_ring(nr, tile, kb, 0, total);
        if (r.stages < (total < 4 ? total : 4) || r.stages > RW_MAX_STAGES || r.smem > RW_SMEM_MAX) return 3;
        // the last k block's rows, as far as the descriptor reads, lie inside the allocation
        if ((r.stages - 1) * r.stage + (kb - 1) * nr * 128 + RW_MMA_ROWS * 128 > r.tail_off) return 4;
      }
  }
  return 0;
}
"""


def test_stages_and_room(tmp_path):
    (tmp_path / "ring.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "ring"), str(tmp_path / "ring.cpp")], check=True)
    assert subprocess.run([str(tmp_path / "ring")]).returncode == 0
