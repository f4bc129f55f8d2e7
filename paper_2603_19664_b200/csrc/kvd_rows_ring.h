// Shared memory of the few-row projection kernel (kvd_rows.cu): its ring of weight and row tiles.  (Plain C++.)
#pragma once

namespace kvd {

constexpr int RW_MAX_ROWS = 64;
constexpr int RW_FEW_ROWS = 16;
constexpr int RW_HEAD_TILE = 32;  // columns per CTA of a key or value head
constexpr int RW_MIN_TILE = 16;   // columns per tile of a plain product, at least
constexpr int RW_MMA_ROWS = 64;   // M of the MMA
constexpr int RW_MAX_STAGES = 16;
constexpr int RW_BARS = 2 * RW_MAX_STAGES + 6;                   // full, empty per stage; tmem_full[2], tmem_empty[2], head, (16-byte multiple)
constexpr int RW_TAIL = RW_BARS * 8 + 32 + RW_MAX_ROWS * 2 * 4;  // barriers, tmem pointer + abort, 1/rms, key scale
constexpr int RW_SMEM_MAX = 232448;
// Key and value heads leave an SM room for two CTAs of the fp32 streaming attention behind them (9 to 18 KB and 16 K registers
// each; the kernel's launch bounds leave the registers), or up to RW_FEW_ROWS rows for one of the tensor-core streaming
// attention (48 KB, 64 in small grids), which take their places beside a CTA of this kernel and wait there
// instead of being started when it ends.  (Beyond RW_FEW_ROWS rows the tensor-core kernel's find the SMs that have no CTA of
// this kernel: 12 to 64 have one.)  Up to RW_FEW_ROWS rows three stages of 8 k blocks do that: projection alone / step
// with attention, us, two, three, four stages and all of an SM's shared memory: Gemma-3-4B layer 1 x 8192 8.8 / 22.3, 7.6 /
// 21.1, 7.4 / 21.4, 7.4 / 24.0; 16 x 2048 8.3 / 38.3, 7.6 / 37.7, -, 7.7 / 40.0; Qwen3-4B layer 8 x 2048 -, 7.1 / 33.6, 7.2 /
// 34.4, 7.2 / 41.0; 16 rows of a 5120-wide layer alone 12.2, 10.9, -, 10.9.  (Stages of 4 and 6 k blocks cost the projection
// 0.8 and 0.4 us.)  Beyond that the stages are as many as fit RW_HEADS_SMEM; all of an SM / this, step: Gemma-3-4B layer 17 x
// 2048 42.3 / 39.8, 40 x 1024 49.6 / 45.5, 64 x 1024 71.0 / 66.3, and the projection alone is no slower (40 rows 11.2 / 10.8).
constexpr int RW_HEADS_STAGES = 3;
constexpr int RW_HEADS_SMEM = 192 * 1024;

// k blocks per stage (a power of two up to 8): stages of 25 to 50 KB.  A stage costs the two single-thread loops some
// 300 clocks of waits and commits whatever it holds (10240 x 2560, one row: 31, 27 and 23 us with 2, 4 and 8), and a plain
// product's ring needs four.  `many`: more than RW_FEW_ROWS rows.
inline int rows_stage_kb(int tile, bool many) {
  int kb = 8;
  while (kb > 1 && kb * (tile + (many ? RW_MAX_ROWS : RW_FEW_ROWS)) * 128 > 50 * 1024) kb /= 2;
  return kb;
}

struct RowsRing {
  int stage, stages, tail_off, smem;  // bytes of a stage, stages, bytes in front of the tail and altogether
};
// Rows padded to `nr`, d_head 0 for a plain product, `total` stages that a CTA fills over all of its tiles.
inline RowsRing rows_ring(int nr, int tile, int stage_kb, int d_head, int total) {
  RowsRing r;
  r.stage = stage_kb * (nr + tile) * 128;
  const int tail = RW_TAIL + (d_head > 0 ? nr * (d_head + 4) * 4 : 0);
  // the descriptor of the last stage's last k block spans RW_MMA_ROWS rows from that block's rows on
  const int beyond = RW_MMA_ROWS * 128 - (r.stage - (stage_kb - 1) * nr * 128), slack = beyond > 0 ? beyond : 0;
  const bool few = nr <= RW_FEW_ROWS;
  int most = d_head > 0 && few ? RW_HEADS_STAGES : RW_MAX_STAGES;
  if (most > total) most = total;
  r.stages = ((d_head > 0 ? RW_HEADS_SMEM : RW_SMEM_MAX) - tail - slack) / r.stage;
  if (r.stages > most) r.stages = most;
  r.tail_off = r.stages * r.stage + slack;
  r.smem = r.tail_off + tail;
  return r;
}

}  // namespace kvd
