// ATTENTION of Algorithm 1 (Eq. 6-7) for many query tokens of one sequence on the fifth-generation tensor cores.
//
//   CTA   = (tile of query tokens, KV head): 128 MMA rows = 128 / G tokens x the G query heads of the head's group (for
//           G = 3, 42 tokens and two empty rows; empty rows are zeros that are never stored).
//   pair  = for d_head 256 two CTAs with neighbouring tiles of the same KV head form a cluster and run the products
//           as tcgen05.mma.cta_group::2 (M = 256, 128 rows per CTA): a K or V block is shared by the pair, each CTA
//           loads and holds half of it (K: half the keys, V: half the channels -- the halves the instruction reads from
//           either shared memory).  Half the bytes per CTA through L2 and shared memory, twice the blocks in flight.
//   keys  = blocks of 64, aligned to ABSOLUTE position, walked in ascending order from the first block any row of the
//           pair can see to the last one.
//   TMEM  = [ O : d_head columns | S_0, S_1 : 64 columns each | Q : d_head / 2 columns ].  The query tile is written
//           there once (two elements per 32-bit column) and is the A operand of S_j = Q K_j^T; the softmax threads
//           read S_j (one row per thread, no shuffles) and hand its columns back at once (scores that are free early
//           let S run two blocks ahead); the weights P_j, in the element type, are the A operand of O += P_j V_j --
//           from 2 x 32 more columns of tensor memory for d_head <= 128, from shared memory at 256, where tensor
//           memory is full.
//   warps = 0-7 softmax and epilogue (two groups of four, TMEM lane quarter = warp % 4, alternating blocks), 8 issues
//           the S products, 9 the PV products (in the pair's leading CTA only), 10-13 gather K/V blocks from the
//           segments with 16-byte cp.async into the 128-byte-swizzled layouts the two products expect (K block:
//           K-major B operand, rows = keys; V block: the same bytes read as an MN-major B operand, rows = the
//           contraction index), a ring of K blocks and a ring of V blocks.  Positions no segment holds are
//           zero-filled and masked.
//   order = S_j is issued as soon as its K block has landed and the softmax threads have read S_{j-2} out of its
//           columns, so the scores run up to two blocks ahead of the softmax; PV_j follows the softmax of block j.  O is
//           rescaled in tensor memory only when a row of the warp moves its reference maximum (the others multiply by
//           exactly 1), and a row moves it only when a block's maximum exceeds it by a factor of 256: with exact maxima
//           some row of a 128-row tile moves in nearly every block, and rescale -> PV_j -> rescale is a serial chain.
//
// A row's result depends on that row alone: the rows of an MMA are computed independently, every row walks the key
// blocks in ascending order, a block without a visible key for the row changes nothing for it (weights 0, rescale by
// exactly 1, O += 0), and the block boundaries are absolute.  So a token attended alone and the same token inside any
// tile give the same bits.  They are not the bits of kvd_decode_attention (another split of the keys, P rounded before
// the second product).  Every wait is bounded: on a timeout the CTA raises the status word, all roles leave their
// loops, and tensor memory is freed.
#include <math_constants.h>
#include <stdlib.h>
#include <string.h>

#include <type_traits>

#include "kvd_internal.h"
#include "kvd_ptx.cuh"

namespace kvd {

constexpr int PT_ROWS = 128;     // MMA rows per CTA
constexpr int PT_KEYS = 64;      // keys per block
constexpr int PT_THREADS = 448;  // fourteen warps
constexpr int PT_LOADERS = 128;  // threads of warps 10-13
constexpr float PT_TAU = 8.0f;   // log2 of the largest weight a row may reach before its reference maximum moves
constexpr int PT_LAG = 3;        // blocks a loader thread keeps in flight behind the one it is issuing

template <int D_HEAD, bool PAIR>
struct PtCfg {
  static constexpr int NCTA = PAIR ? 2 : 1;
  static constexpr int LOADERS = PT_LOADERS;
  static constexpr int K_ROWS = PT_KEYS / NCTA;                   // keys of a block this CTA holds
  static constexpr int V_COLS = D_HEAD / NCTA;                    // channels of a block this CTA holds
  static constexpr int TILE_BYTES = PT_KEYS * D_HEAD * 2 / NCTA;  // this CTA's share of one K or V block
  static constexpr int SLAB_K = K_ROWS * 128;                     // 64 channels of this CTA's keys
  static constexpr int SLAB_V = PT_KEYS * 128;                    // 64 of this CTA's channels of every key
  static constexpr int SLOTS_K = D_HEAD == 256 ? (PAIR ? 6 : 3) : (PAIR ? 6 : 4);  // blocks in the K ring (the scores run ahead)
  static constexpr int SLOTS_V = D_HEAD == 256 ? (PAIR ? 4 : 2) : (PAIR ? 6 : 4);  // blocks in the V ring
  static constexpr int SLOTS = SLOTS_K + SLOTS_V;
  static constexpr int COL_O = 0, COL_S = D_HEAD, COL_Q = D_HEAD + 2 * PT_KEYS;
  static constexpr bool P_TMEM = D_HEAD <= 128;                   // room for the weights in tensor memory as well
  static constexpr int COL_P = COL_Q + D_HEAD / 2;                // two blocks of weights, 32 columns each (P_TMEM)
  static constexpr int COLS_USED = COL_P + (P_TMEM ? PT_KEYS : 0);
  static constexpr int COLS = COLS_USED <= 256 ? 256 : 512;       // allocation: a power of two
  static constexpr int P_BYTES = P_TMEM ? 0 : PT_ROWS * PT_KEYS * 2;  // one block of weights in shared memory otherwise
  static constexpr int N_BARS = 2 * SLOTS + 22;
  static constexpr int SMEM_BYTES = 1024 + SLOTS * TILE_BYTES + 2 * P_BYTES + N_BARS * 8;
};

// A wait of this kernel.  Every SM sub-partition hosts a warp of either softmax group, a loader warp and possibly an MMA
// thread, and at any time some of them wait: a short sleep between polls leaves the issue slots to the warps that
// compute (+2 to 7 %).  CLUSTER: the barrier may be completed by the partner CTA, by its threads' arrivals or by bytes that
// it sends (st.async, bulk copies).  Both release at cluster scope, and only an acquire of that scope synchronises with
// them.  (A commit of the pair's products needs none: what it announces lies in this CTA's tensor memory or rings and is
// ordered by tcgen05.fence.)
template <bool CLUSTER>
__device__ __forceinline__ bool polite_wait(uint32_t bar, uint32_t parity, const volatile int *abort_flag, unsigned long long timeout_ns) {
  auto done = [&]() { return CLUSTER ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (done()) return true;
  const unsigned long long t0 = globaltimer_ns();
  uint32_t it = 0;
  while (!done()) {
    __nanosleep(20);
    if (((++it) & 31u) == 0u && (*abort_flag != 0 || globaltimer_ns() - t0 > timeout_ns)) return false;
  }
  return true;
}
// The same for a whole warp.  Every lane asks once, and usually that is all: with lane 0 asking alone behind a branch and
// handing the answer on, a wait for a barrier that had long completed took a softmax warp 200 to 290 clocks.  Otherwise
// lane 0 waits, and the result is broadcast.
template <bool CLUSTER = false>
__device__ __forceinline__ bool polite_warp_wait(uint32_t bar, uint32_t parity, const volatile int *abort_flag, unsigned long long timeout_ns, int lane) {
  if (__all_sync(0xffffffffu, CLUSTER ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity))) return true;
  int ok = 1;
  if (lane == 0) ok = polite_wait<CLUSTER>(bar, parity, abort_flag, timeout_ns) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();  // the other lanes' reads follow lane 0's acquire
  return ok != 0;
}
template <bool PAIR>
__device__ __forceinline__ bool lead_wait(uint32_t bar, uint32_t parity, const volatile int *abort_flag, unsigned long long timeout_ns) {
  return polite_wait<PAIR>(bar, parity, abort_flag, timeout_ns);
}

// The kernels are programmatic dependents of what precedes them: up to here (barriers, tensor memory) they may run while it
// ends.  Their own dependents are let in after the allocation, which waits without a limit.
__device__ __forceinline__ void early_start_point() {
  grid_launch_dependents();
  grid_dependency_wait();
}

// Whether every row of a warp sees every key of a block, without the row's masks (which cost 460 of the 2380 clocks a
// softmax warp took for a block): the block lies inside one segment and inside the range all the warp's rows see.
// Rows that are not stored do not count.
struct PtWhole {
  int lo, hi;         // the range that every stored row of the warp sees
  int seg0, seg_len;  // the segment the last block was found in
  __device__ __forceinline__ PtWhole(bool valid, int row_lo, int row_hi) : seg0(0), seg_len(0) {
    lo = __reduce_max_sync(0xffffffffu, valid ? row_lo : INT_MIN);
    hi = __reduce_min_sync(0xffffffffu, valid ? row_hi : INT_MAX);
  }
  __device__ __forceinline__ bool operator()(const PrefillParams &P, int pos0) {
    if (pos0 < lo || pos0 + PT_KEYS - 1 > hi) return false;
    if (!segment_holds(seg0, seg_len, pos0, PT_KEYS)) {
#pragma unroll
      for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg)
        if (segment_holds(P.first[sg], P.len[sg], pos0, 1)) {
          seg0 = P.first[sg];
          seg_len = P.len[sg];
        }
    }
    return segment_holds(seg0, seg_len, pos0, PT_KEYS);
  }
};
// Which keys of the block at pos0 does a row see: present in a segment, in [lo, qp] (bit k = key pos0 + k).
__device__ __forceinline__ unsigned long long pt_visible(const PrefillParams &P, int pos0, int lo, int qp) {
  unsigned long long vis = 0ull;
#pragma unroll
  for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg) vis |= segment_slots(P.first[sg], P.len[sg], pos0);
  return vis & visible_slots(lo, qp, pos0);
}
// Scores of invisible keys become -inf; the maximum of the 64 in four chains of three-input maxima.
__device__ __forceinline__ float pt_mask_max(uint32_t (&s0)[32], uint32_t (&s1)[32], bool whole, unsigned long long vis) {
  if (!whole) {
    const uint32_t v0 = static_cast<uint32_t>(vis), v1 = static_cast<uint32_t>(vis >> 32);
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if (!((v0 >> k) & 1u)) s0[k] = 0xff800000u;  // -inf
      if (!((v1 >> k) & 1u)) s1[k] = 0xff800000u;
    }
  }
  float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
  for (int k = 0; k < 32; k += 8) {
    mx[0] = fmax3(mx[0], __uint_as_float(s0[k]), __uint_as_float(s0[k + 1]));
    mx[1] = fmax3(mx[1], __uint_as_float(s0[k + 2]), __uint_as_float(s0[k + 3]));
    mx[2] = fmax3(mx[2], __uint_as_float(s0[k + 4]), __uint_as_float(s0[k + 5]));
    mx[3] = fmax3(mx[3], __uint_as_float(s0[k + 6]), __uint_as_float(s0[k + 7]));
    mx[0] = fmax3(mx[0], __uint_as_float(s1[k]), __uint_as_float(s1[k + 1]));
    mx[1] = fmax3(mx[1], __uint_as_float(s1[k + 2]), __uint_as_float(s1[k + 3]));
    mx[2] = fmax3(mx[2], __uint_as_float(s1[k + 4]), __uint_as_float(s1[k + 5]));
    mx[3] = fmax3(mx[3], __uint_as_float(s1[k + 6]), __uint_as_float(s1[k + 7]));
  }
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}
// Weights 2^(s * scale - m) of 64 scores: two per fused multiply-add; the row sum adds them up in fp32, the product
// takes them rounded to the element type.
template <int DT>
__device__ __forceinline__ void pt_weights(const uint32_t (&s0)[32], const uint32_t (&s1)[32], uint64_t c2, uint64_t nm2, uint64_t (&l2)[2],
                                           uint32_t (&w)[32]) {
  const uint64_t one2 = pack2(1.0f, 1.0f);
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    float e0, e1;
    unpack2(ffma2(pack2(__uint_as_float(s0[k]), __uint_as_float(s0[k + 1])), c2, nm2), e0, e1);
    const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);
    w[k >> 1] = pack_out<DT>(p0, p1);
    l2[(k >> 1) & 1] = ffma2(pack2(p0, p1), one2, l2[(k >> 1) & 1]);
  }
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    float e0, e1;
    unpack2(ffma2(pack2(__uint_as_float(s1[k]), __uint_as_float(s1[k + 1])), c2, nm2), e0, e1);
    const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);
    w[16 + (k >> 1)] = pack_out<DT>(p0, p1);
    l2[(k >> 1) & 1] = ffma2(pack2(p0, p1), one2, l2[(k >> 1) & 1]);
  }
}
// A part of the row sum, referred to another maximum.  The factor goes to the four chains, as in a further block
// without a visible key: whether the tile has such blocks behind the row's last one must not show in the row's bits.
__device__ __forceinline__ float pt_row_sum(const uint64_t (&l2)[2], float factor) {
  const uint64_t f2 = pack2(factor, factor);
  float a0, a1, a2, a3;
  unpack2(fmul2(l2[0], f2), a0, a1);
  unpack2(fmul2(l2[1], f2), a2, a3);
  return (a0 + a1) + (a2 + a3);
}
// O (D_HEAD columns of this warp's lanes, from column `col`) times a factor per row.
template <int D_HEAD>
__device__ __forceinline__ void pt_rescale(uint32_t col, float alpha) {
#pragma unroll 1
  for (int c = 0; c < D_HEAD / 32; ++c) {
    uint32_t r[32];
    tmem_ld_x32(col + c * 32, r);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
    tmem_st_x32(col + c * 32, r);
  }
  tmem_wait_st();
}

// The loader warps of a CTA: K and V blocks blk0 .. blk0 + n_blk - 1 of KV head kvh into the rings.
template <class Cfg, int D_HEAD, class Arrive>
__device__ __forceinline__ void pt_load_blocks(const PrefillParams &P, uint32_t ring, uint32_t ring_v, uint32_t bar_base, int slots, int blk0, int n_blk,
                                               int kvh, int rank, int ptid, const Arrive &arrive_lead, volatile int *s_abort,
                                               unsigned long long tmo) {
  constexpr int SLOTS_K = Cfg::SLOTS_K, SLOTS_V = Cfg::SLOTS_V;
  const int lane = ptid & 31;
  auto bar_full = [&](int v, int sl) { return bar_base + 8u * (v * SLOTS_K + sl); };
  auto bar_empty = [&](int v, int sl) { return bar_base + 8u * (slots + v * SLOTS_K + sl); };
  // ------------------------------------------------------------------ K/V blocks into the rings
  // issue order = the order the products want them, the keys three blocks ahead: K_0 K_1 K_2 | K_3 V_0 | K_4 V_1 | ...
  // This CTA's share of a block: K_ROWS keys of all channels (K), all 64 keys of V_COLS channels (V).
  // blocks issued and not yet published to the MMA threads, oldest first.  A block is published once PT_LAG younger
  // ones have been issued -- or at once, all of them, when the next block would have to wait for a free slot (the
  // slot is freed by a product that may itself be waiting for one of these blocks).
  uint32_t pend[PT_LAG + 1] = {};
  int n_pend = 0;
  bool ok = true;
  auto publish_all = [&]() {
    cp_async_wait_all();
    fence_proxy_async_smem();
    __syncwarp();
#pragma unroll
    for (int i = 0; i <= PT_LAG; ++i)
      if (i < n_pend && lane == 0) arrive_lead(pend[i]);
    n_pend = 0;
  };
  // rows [row_first, row_first + ROWS) of the block, CPR 16-byte pieces of each starting at element col_first
  auto gather = [&](auto rows_c, auto cpr_c, uint32_t base, int slab_bytes, int pos_first, int col_first, bool is_v) {
    constexpr int ROWS = decltype(rows_c)::value, CPR = decltype(cpr_c)::value;
    constexpr int RSTEP = Cfg::LOADERS / CPR;  // rows one pass of the loader threads covers
    const int c = ptid % CPR, r0 = ptid / CPR;
    const uint32_t dst = base + static_cast<uint32_t>(c >> 3) * slab_bytes;
    // the usual case: one segment holds all the rows -> one base pointer, one stride
    int whole = -1;
#pragma unroll
    for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg)
      if (segment_holds(P.first[sg], P.len[sg], pos_first, ROWS)) whole = sg;
    if (whole >= 0) {
      const long long stride = P.stride[whole];
      const __nv_bfloat16 *src = (is_v ? P.v[whole] : P.k[whole]) + static_cast<size_t>(pos_first - P.first[whole] + r0) * stride +
                                 static_cast<size_t>(kvh) * D_HEAD + col_first + c * 8;
#pragma unroll
      for (int pass = 0; pass < ROWS / RSTEP; ++pass) {
        const int r = r0 + pass * RSTEP;
        cp_async16(dst + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, true);
        src += RSTEP * stride;
      }
    } else {
#pragma unroll 1
      for (int pass = 0; pass < ROWS / RSTEP; ++pass) {
        const int r = r0 + pass * RSTEP, pos = pos_first + r;
        const __nv_bfloat16 *src = P.q;
        bool have = false;
#pragma unroll
        for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg) {
          const int rr = pos - P.first[sg];
          if (rr >= 0 && rr < P.len[sg]) {
            src = (is_v ? P.v[sg] : P.k[sg]) + static_cast<size_t>(rr) * P.stride[sg] + static_cast<size_t>(kvh) * D_HEAD + col_first + c * 8;
            have = true;
          }
        }
        cp_async16(dst + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, have);
      }
    }
  };
  auto emit = [&](int is_v, int j) -> bool {
    const int n_slots = is_v ? SLOTS_V : SLOTS_K, slot = j % n_slots;
    if (j >= n_slots) {
      const uint32_t par = ((j / n_slots) - 1) & 1;
      int free_now = lane == 0 ? (mbar_try_wait(bar_empty(is_v, slot), par) ? 1 : 0) : 0;
      free_now = __shfl_sync(0xffffffffu, free_now, 0);
      if (!free_now) {
        publish_all();
        int got = lane == 0 ? (polite_wait<false>(bar_empty(is_v, slot), par, s_abort, tmo) ? 1 : 0) : 0;
        got = __shfl_sync(0xffffffffu, got, 0);
        if (!got) return false;
      }
    }
    const int pos0 = (blk0 + j) * PT_KEYS;
    if (is_v)
      gather(std::integral_constant<int, PT_KEYS>(), std::integral_constant<int, Cfg::V_COLS / 8>(), ring_v + slot * Cfg::TILE_BYTES,
             Cfg::SLAB_V, pos0, static_cast<int>(rank) * Cfg::V_COLS, true);
    else
      gather(std::integral_constant<int, Cfg::K_ROWS>(), std::integral_constant<int, D_HEAD / 8>(), ring + slot * Cfg::TILE_BYTES,
             Cfg::SLAB_K, pos0 + static_cast<int>(rank) * Cfg::K_ROWS, 0, false);
    cp_async_commit();
#pragma unroll
    for (int i = 0; i <= PT_LAG; ++i)
      if (i == n_pend) pend[i] = bar_full(is_v, slot);
    ++n_pend;
    if (n_pend > PT_LAG) {
      // the oldest block has PT_LAG younger ones behind it: it has landed by now, or nearly
      cp_async_wait_group<PT_LAG>();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) arrive_lead(pend[0]);
#pragma unroll
      for (int i = 0; i < PT_LAG; ++i) pend[i] = pend[i + 1];
      --n_pend;
    }
    return true;
  };
  if (n_blk > 0) {
    ok = emit(0, 0);
    if (ok && n_blk > 1) ok = emit(0, 1);
    if (ok && n_blk > 2) ok = emit(0, 2);
    for (int j = 0; ok && j < n_blk; ++j) {
      if (j + 3 < n_blk) ok = emit(0, j + 3);
      if (ok) ok = emit(1, j);
    }
    if (ok) publish_all();
    else {
      cp_async_wait_all();
      raise(P.status, STATUS_TIMEOUT, s_abort);
    }
  }
}

template <int D_HEAD, int G, int DT, bool PAIR>
__global__ void __launch_bounds__(PT_THREADS, 1) kvd_prefill_attn_tc_kernel(const __grid_constant__ PrefillParams P) {
  using Cfg = PtCfg<D_HEAD, PAIR>;
  constexpr int TOK = PT_ROWS / G;     // query tokens per CTA (G = 3: 42 tokens, the last two MMA rows stay empty)
  constexpr int NCTA = Cfg::NCTA;
  constexpr int SLOTS = Cfg::SLOTS, SLOTS_K = Cfg::SLOTS_K, SLOTS_V = Cfg::SLOTS_V;
  extern __shared__ uint8_t pt_smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort_i, s_lo, s_hi;
  __shared__ float s_mx[2][PT_ROWS], s_lx[2][PT_ROWS];  // per group: the row maximum after its last block, its part of the row sum
  volatile int *s_abort = &s_abort_i;
  // the rings start on a 1024-byte boundary (the swizzle is a function of the address), the barriers follow them
  const uint32_t ring = (smem_u32(pt_smem_raw) + 1023u) & ~1023u;
  const uint32_t ring_v = ring + SLOTS_K * Cfg::TILE_BYTES;  // K blocks first, V blocks behind them
  const uint32_t p_smem = ring + SLOTS * Cfg::TILE_BYTES;    // two blocks of weights
  const uint32_t bar_base = p_smem + 2 * Cfg::P_BYTES;
  // barriers the MMA threads wait on are used in the leading CTA only; the others (MMA commits) in both
  auto bar_full = [&](int v, int s) { return bar_base + 8u * (v * SLOTS_K + s); };           // leader: a block has landed
  auto bar_empty = [&](int v, int s) { return bar_base + 8u * (SLOTS + v * SLOTS_K + s); };  // both: its product is done
  auto bar_s_full = [&](int b) { return bar_base + 8u * (2 * SLOTS + b); };                  // both: scores of a block
  auto bar_p_ready = [&](int b) { return bar_base + 8u * (2 * SLOTS + 2 + b); };             // leader: weights in place
  auto bar_pv_done = [&](int b) { return bar_base + 8u * (2 * SLOTS + 4 + b); };             // both: O += P V finished
  const uint32_t bar_o_full = bar_base + 8u * (2 * SLOTS + 6), bar_q_ready = bar_base + 8u * (2 * SLOTS + 7);
  auto bar_s_free = [&](int b) { return bar_base + 8u * (2 * SLOTS + 8 + b); };              // leader: scores were read
  auto bar_m = [&](int grp, int q) { return bar_base + 8u * (2 * SLOTS + 10 + grp * 4 + q); };  // own: a row maximum was handed over
  auto bar_l = [&](int q) { return bar_base + 8u * (2 * SLOTS + 18 + q); };                     // own: both parts of the row sums

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  // One-dimensional grid in the order the CTAs should start: long tiles (late tokens of a causal call) first, and for
  // every tile (pair of neighbouring tiles) all KV heads before the next shorter one -- with the heads as a second grid
  // dimension the longest tiles of the last head would start last and set the launch's length.
  const int n_tiles = static_cast<int>(gridDim.x) / P.n_kv;        // even for pairs
  const int slot = static_cast<int>(blockIdx.x) / NCTA;            // cluster (or CTA) in start order
  const int kvh = slot % P.n_kv;
  const int tile = n_tiles - 1 - ((slot / P.n_kv) * NCTA + static_cast<int>(blockIdx.x) % NCTA);
  const int tok0 = tile * TOK;
  const int pair_tok0 = PAIR ? (tile & ~1) * TOK : tok0;           // tiles 2c and 2c + 1 share a cluster
  const unsigned long long tmo = P.timeout_ns;
  // An arrival of one warp on a barrier of the leading CTA.  Across the pair it is a relaxed arrive: what it announces
  // (scores read out of tensor memory; weights or K/V pieces written to this CTA's own shared memory) has been
  // completed and fenced for the tensor cores' proxy by the announcing threads before they get here, and a
  // cluster-scope release would make the warp wait for every outstanding memory operation of a busy SM.
  auto arrive_lead = [&](uint32_t bar) {
    if (!PAIR || rank == 0) mbar_arrive(bar);
    else mbar_arrive_cluster(map_to_cta(bar, 0));
  };

  if (tid == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(bar_full(0, s), 4 * NCTA);  // one arrival per loader warp of the pair
      mbar_init(bar_empty(0, s), 1);        // the MMA commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_s_full(b), 1);          // the MMA commit
      mbar_init(bar_p_ready(b), 4 * NCTA);  // one arrival per softmax warp of the group, in both CTAs
      mbar_init(bar_pv_done(b), 1);
      mbar_init(bar_s_free(b), 4 * NCTA);   // the same
    }
    for (int q = 0; q < 4; ++q) {
      mbar_init(bar_m(0, q), 1);  // the warp of the group that owns these 32 rows
      mbar_init(bar_m(1, q), 1);
      mbar_init(bar_l(q), 2);     // that warp of either group
    }
    mbar_init(bar_o_full, 1);
    mbar_init(bar_q_ready, 8 * NCTA);
    fence_mbar_init();
    s_abort_i = 0;
    s_lo = INT_MAX;
    s_hi = -1;
  }
  if (warp == 8) {
    if constexpr (PAIR) {
      tmem_alloc_pair(smem_u32(&s_tmem), Cfg::COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(&s_tmem), Cfg::COLS);
      tmem_relinquish();
    }
  }
  __syncthreads();
  early_start_point();
  // ---- key positions the pair needs: from the smallest first-visible to the largest last-visible of its tokens
  if (tid < NCTA * TOK && pair_tok0 + tid < P.n_rows) {
    const int qp = P.q_pos[pair_tok0 + tid];
    int lo = first_visible(qp, P.window);
    lo = lo < P.seg_lo ? P.seg_lo : lo;
    const int hi = qp < P.seg_hi ? qp : P.seg_hi;
    if (hi >= lo) {
      atomicMin(&s_lo, lo);
      atomicMax(&s_hi, hi);
    }
  }
  tc_fence_before();
  if constexpr (PAIR) cluster_sync_all();  // barriers of both CTAs are initialised before anyone signals across the pair
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = s_tmem;
  const int blk0 = s_hi >= 0 ? s_lo / PT_KEYS : 0;
  const int n_blk = s_hi >= 0 ? s_hi / PT_KEYS - blk0 + 1 : 0;

  if (warp < 8) {
    // ------------------------------------------------------------------ softmax and epilogue: thread = MMA row
    // two warpgroups share the 128 rows: group 0 takes the even blocks, group 1 the odd ones, each with its own score
    // and weight buffer.  What a row carries from block to block is its running maximum, handed from group to group
    // through shared memory; every group keeps its own part of the row sum.
    const int wg = warp >> 2, q4 = warp & 3;
    const int row = q4 * 32 + lane;
    const int tok = tok0 + row / G, g = row % G;
    const bool valid = row / G < TOK && tok < P.n_rows;
    const int qp = valid ? P.q_pos[tok] : -1;
    const int lo = first_visible(qp, P.window);
    const uint32_t lane_field = static_cast<uint32_t>(q4 * 32) << 16;
    const size_t row_off = (static_cast<size_t>(valid ? tok : 0) * P.n_q + kvh * G + (valid ? g : 0)) * D_HEAD;
    if (n_blk > 0) {
      // the query row into tensor memory: element pairs (2c, 2c + 1) -> column c (zeros for padding rows)
      const uint4 *qsrc = reinterpret_cast<const uint4 *>(P.q + row_off);
#pragma unroll 1
      for (int c = wg; c < D_HEAD / 64; c += 2) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 w = valid ? qsrc[c * 8 + i] : make_uint4(0u, 0u, 0u, 0u);
          r[4 * i] = w.x;
          r[4 * i + 1] = w.y;
          r[4 * i + 2] = w.z;
          r[4 * i + 3] = w.w;
        }
        tmem_st_x32(tmem_base + lane_field + Cfg::COL_Q + c * 32, r);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_lead(bar_q_ready);
    }
    float m_own = -CUDART_INF_F;    // the maximum this group's part of the row sum refers to
    uint64_t l2[2] = {0ull, 0ull};  // that part, in four chains (two packed pairs)
    bool ok = true;
    const uint64_t c2 = pack2(P.scale_log2e, P.scale_log2e);
    PtWhole whole_block(valid, lo, qp);
    const int buf = wg;
    for (int j = wg; j < n_blk; j += 2) {
      const uint32_t ph = (j >> 1) & 1;
      if (!polite_warp_wait(bar_s_full(buf), ph, s_abort, tmo, lane)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t s_col = tmem_base + lane_field + Cfg::COL_S + buf * PT_KEYS;
      uint32_t s0[32], s1[32];
      tmem_ld_x32(s_col, s0);
      tmem_ld_x32(s_col + 32, s1);
      const bool whole = whole_block(P, (blk0 + j) * PT_KEYS);  // (warp-uniform)
      unsigned long long vis = ~0ull;
      if (!whole) vis = pt_visible(P, (blk0 + j) * PT_KEYS, lo, qp);
      tmem_wait_ld();
      // the scores are in registers: their columns may take this group's next block
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_lead(bar_s_free(buf));
      const float bm = pt_mask_max(s0, s1, whole, vis) * P.scale_log2e;  // log2 units (scale > 0)
      // the row's maximum after block j - 1 comes from the other group; the one after block j goes back to it
      float m_prev = -CUDART_INF_F;
      if (j > 0) {
        if (!polite_warp_wait(bar_m(wg ^ 1, q4), ((j - 1) >> 1) & 1, s_abort, tmo, lane)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
          break;
        }
        m_prev = s_mx[wg ^ 1][row];
      }
      // The reference m the weights 2^(s - m) are taken against follows the row's maximum lazily: it moves (and O and
      // the row sums are rescaled) only when a block's maximum exceeds it by more than 2^PT_TAU; until then the
      // weights may reach 2^PT_TAU, which fp32 sums and 16-bit weights hold as well as values below 1.  A function of
      // the row's own scores and of the block order alone, like the maximum itself.
      const float m_new = m_prev == -CUDART_INF_F ? bm : (bm > m_prev + PT_TAU ? bm : m_prev);
      s_mx[wg][row] = m_new;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_m(wg, q4));
      const float m_use = m_new == -CUDART_INF_F ? 0.f : m_new;
      // rescale of what the row has so far: exactly 1 when its maximum stays; while nothing has been seen O and l are 0
      const float alpha = m_prev == -CUDART_INF_F ? 1.0f : ex2_approx(m_prev - m_use);
      const float alpha_own = m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use);
      m_own = m_new;
      uint32_t w[32];
      const uint64_t al2 = pack2(alpha_own, alpha_own);
      l2[0] = fmul2(l2[0], al2);
      l2[1] = fmul2(l2[1], al2);
      pt_weights<DT>(s0, s1, c2, pack2(-m_use, -m_use), l2, w);
      // P_j into shared memory as a K-major A operand (row = MMA row, 128 bytes = 64 keys, 128-byte swizzle); the
      // product that read this buffer two blocks ago has long finished
      if (j >= 2 && !polite_warp_wait(bar_pv_done(buf), ((j - 2) >> 1) & 1, s_abort, tmo, lane)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
        break;
      }
      if constexpr (Cfg::P_TMEM) {
        tmem_st_x32(tmem_base + lane_field + Cfg::COL_P + buf * (PT_KEYS / 2), w);
      } else {
        const uint32_t prow = p_smem + buf * Cfg::P_BYTES + row * 128;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(prow + ((i ^ (row & 7)) << 4)), "r"(w[4 * i]), "r"(w[4 * i + 1]),
                       "r"(w[4 * i + 2]), "r"(w[4 * i + 3])
                       : "memory");
        fence_proxy_async_smem();
      }
      if (__any_sync(0xffffffffu, alpha != 1.0f)) {
        // O holds the blocks before j; the last of those products must have finished (j >= 1 here: a maximum exists)
        if (!polite_warp_wait(bar_pv_done(buf ^ 1), ((j - 1) >> 1) & 1, s_abort, tmo, lane)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
          break;
        }
        tc_fence_after();
        pt_rescale<D_HEAD>(tmem_base + lane_field + Cfg::COL_O, alpha);
        tc_fence_before();
      } else if constexpr (Cfg::P_TMEM) {
        tmem_wait_st();
        tc_fence_before();
      }
      __syncwarp();
      if (lane == 0) arrive_lead(bar_p_ready(buf));
    }
    // ---- the row sum: both parts referred to the final maximum, added in group order
    float l_run = 0.f;
    if (ok && n_blk > 0) {
      const int last = n_blk - 1;
      float m_fin = m_own;
      if ((last & 1) != wg) {
        if (!polite_warp_wait(bar_m(wg ^ 1, q4), (last >> 1) & 1, s_abort, tmo, lane)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
        }
        m_fin = s_mx[wg ^ 1][row];
      }
      if (ok) {
        const float m_use = m_fin == -CUDART_INF_F ? 0.f : m_fin;
        s_lx[wg][row] = pt_row_sum(l2, m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use));
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_l(q4));
        if (!polite_warp_wait(bar_l(q4), 0, s_abort, tmo, lane)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
        }
        l_run = s_lx[0][row] + s_lx[1][row];
      }
    }
    // ---- normalise and store, each group its half of the channels (a token without a visible key yields zeros)
    if (ok && n_blk > 0 && !polite_warp_wait(bar_o_full, 0, s_abort, tmo, lane)) {
      raise(P.status, STATUS_TIMEOUT, s_abort);
      ok = false;
    }
    if (ok) {
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
      uint4 *dst = reinterpret_cast<uint4 *>(P.out + row_off);
#pragma unroll 1
      for (int c = wg * (D_HEAD / 64); c < (wg + 1) * (D_HEAD / 64); ++c) {
        uint32_t r[32];
        if (n_blk > 0) {
          tmem_ld_x32(tmem_base + lane_field + Cfg::COL_O + c * 32, r);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
        }
        uint32_t o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = pack_out<DT>(__uint_as_float(r[2 * i]) * inv, __uint_as_float(r[2 * i + 1]) * inv);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 4; ++i) dst[c * 4 + i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
        }
      }
    }
  } else if (warp == 8 || warp == 9) {
    // ------------------------------------------------------------------ MMA issue (one thread per product, leading CTA)
    constexpr uint32_t IDESC_BASE = (DT == 0 ? umma_idesc_bf16_f32(PT_ROWS * NCTA, 8) : umma_idesc_f16_f32(PT_ROWS * NCTA, 8)) & ~(1u << 17);
    constexpr uint32_t IDESC_S = IDESC_BASE | (static_cast<uint32_t>(PT_KEYS >> 3) << 17);              // N = 64 keys, B K-major
    constexpr uint32_t IDESC_O = IDESC_BASE | (static_cast<uint32_t>(D_HEAD >> 3) << 17) | (1u << 16);  // N = d_head, B MN-major
    auto commit = [&](uint32_t bar) {
      if constexpr (PAIR) umma_commit_pair(bar, 3);  // the barrier at this offset in both CTAs
      else umma_commit(bar);
    };
    if (lane == 0 && n_blk > 0 && rank == 0 && warp == 8) {
      // S_j = Q K_j^T into score buffer j & 1, as far ahead of the softmax as the two buffers allow
      bool ok = lead_wait<PAIR>(bar_q_ready, 0, s_abort, tmo);
      tc_fence_after();
      for (int j = 0; ok && j < n_blk; ++j) {
        const int slot = j % SLOTS_K;
        // the K block has landed; the softmax threads have read the scores of block j - 2 out of these columns
        if (!lead_wait<PAIR>(bar_full(0, slot), (j / SLOTS_K) & 1, s_abort, tmo) ||
            (j >= 2 && !lead_wait<PAIR>(bar_s_free(j & 1), ((j - 2) >> 1) & 1, s_abort, tmo))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem_base + Cfg::COL_S + (j & 1) * PT_KEYS;
        const uint64_t desc0 = umma_smem_desc_sw128(ring + slot * Cfg::TILE_BYTES);
#pragma unroll
        for (int ks = 0; ks < D_HEAD / 16; ++ks) {
          const uint64_t bdesc = desc0 + (((ks >> 2) * Cfg::SLAB_K + (ks & 3) * 32) >> 4);
          if constexpr (PAIR) umma_f16_ts_pair(d, tmem_base + Cfg::COL_Q + ks * 8, bdesc, IDESC_S, ks > 0 ? 1u : 0u);
          else umma_f16_ts(d, tmem_base + Cfg::COL_Q + ks * 8, bdesc, IDESC_S, ks > 0 ? 1u : 0u);
        }
        commit(bar_empty(0, slot));
        commit(bar_s_full(j & 1));
      }
      if (!ok) raise(P.status, STATUS_TIMEOUT, s_abort);
    } else if (lane == 0 && n_blk > 0 && rank == 0) {
      // O += P_j V_j once the weights are in place (and O has been rescaled where a reference maximum moved)
      bool ok = true;
      for (int j = 0; j < n_blk; ++j) {
        const int slot = j % SLOTS_V;
        if (!lead_wait<PAIR>(bar_p_ready(j & 1), (j >> 1) & 1, s_abort, tmo) ||
            !lead_wait<PAIR>(bar_full(1, slot), (j / SLOTS_V) & 1, s_abort, tmo)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t desc0 = umma_smem_desc_sw128_mn(ring_v + slot * Cfg::TILE_BYTES, Cfg::SLAB_V);
        const uint64_t pdesc0 = umma_smem_desc_sw128(p_smem + (j & 1) * Cfg::P_BYTES);
        const uint32_t ptmem = tmem_base + Cfg::COL_P + (j & 1) * (PT_KEYS / 2);
#pragma unroll
        for (int ks = 0; ks < PT_KEYS / 16; ++ks) {
          const uint64_t vdesc = desc0 + ((ks * 16 * 128) >> 4);
          const uint32_t acc = (j > 0 || ks > 0) ? 1u : 0u;
          if constexpr (Cfg::P_TMEM) {
            if constexpr (PAIR) umma_f16_ts_pair(tmem_base + Cfg::COL_O, ptmem + ks * 8, vdesc, IDESC_O, acc);
            else umma_f16_ts(tmem_base + Cfg::COL_O, ptmem + ks * 8, vdesc, IDESC_O, acc);
          } else {
            if constexpr (PAIR) umma_bf16_pair(tmem_base + Cfg::COL_O, pdesc0 + ((ks * 32) >> 4), vdesc, IDESC_O, acc);
            else umma_bf16(tmem_base + Cfg::COL_O, pdesc0 + ((ks * 32) >> 4), vdesc, IDESC_O, acc);
          }
        }
        commit(bar_empty(1, slot));
        commit(bar_pv_done(j & 1));
      }
      if (ok) commit(bar_o_full);
      else raise(P.status, STATUS_TIMEOUT, s_abort);
    }
  } else {
    pt_load_blocks<Cfg, D_HEAD>(P, ring, ring_v, bar_base, SLOTS, blk0, n_blk, kvh, static_cast<int>(rank), tid - 10 * 32, arrive_lead, s_abort, tmo);
  }

  // ---- teardown: every role is done with tensor memory; in a pair nobody leaves while the partner can still signal
  // into this CTA's shared memory
  tc_fence_before();
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem_base, Cfg::COLS);
    else tmem_dealloc(tmem_base, Cfg::COLS);
  }
}

// ------------------------------------------------------------------------------------------------
// Two row tiles per CTA (d_head 128), for launches that fill the GPU.  In the kernel above the two softmax groups
// take turns on the blocks of one tile, hand the reference maximum to each other in every block and wait for it (and
// for the scores) about a third of the time.  Here each group has a tile of its own, so nothing is exchanged, a K or V
// block is loaded once for 256 rows, and each tile's next scores are there before its softmax asks for them.  A CTA
// takes longer per block than above (1950 against 1550 clocks, for twice the rows), hence only where there are enough
// of them (prefill_dual_pays).  One / two tiles per CTA, Qwen3-4B layer: 4096 tokens 198 / 151 us.
//   TMEM = [ O_0, O_1 : d_head columns each | S_00, S_01, S_10, S_11 : 64 columns each (tile, block parity) ]; the
//          weights of a block overwrite the first half of its scores.  The query tiles are in shared memory.
//   warps = 0-3 tile 0, 4-7 tile 1, 8 and 9 the products of tiles 0 and 1, 10 and 11 loaders: twelve warps leave a
//          thread 168 registers (with four loader warps 128, and spills: 169 instead of 161 us).
//   order = per tile S_0 S_1 | PV_0 S_2 | PV_1 S_3 | ...: one thread issues both products; S_{j+2}, which overwrites the
//          weights of block j, once PV_j has finished.  (Weights in columns of their own next to one score buffer
//          measured no better: 174 us.)
// The bits are those of the kernel above: same blocks, same reference maxima, same products, and the row sum is kept
// in two parts (even and odd blocks), each with the reference it had two blocks ago.
template <int D_HEAD>
struct PdCfg {
  static constexpr int NCTA = 1;
  static constexpr int LOADERS = 64, THREADS = 384;
  static constexpr int K_ROWS = PT_KEYS, V_COLS = D_HEAD;
  static constexpr int TILE_BYTES = PT_KEYS * D_HEAD * 2;
  static constexpr int SLAB_K = PT_KEYS * 128, SLAB_V = PT_KEYS * 128;
  static constexpr int SLAB_Q = PT_ROWS * 128;                   // 64 channels of a query tile
  static constexpr int Q_BYTES = PT_ROWS * D_HEAD * 2;
  static constexpr int SLOTS_K = 5, SLOTS_V = 5, SLOTS = SLOTS_K + SLOTS_V;
  static constexpr int COL_S = 2 * D_HEAD, COLS = 512;
  static constexpr int N_BARS = 2 * SLOTS + 14;                  // + s_full[2][2], p_ready[2][2], pv_done[2], o_full[2], q_ready[2]
  static constexpr int SMEM_BYTES = 1024 + 2 * Q_BYTES + SLOTS * TILE_BYTES + N_BARS * 8;
  static_assert(COL_S + 4 * PT_KEYS <= COLS && SMEM_BYTES <= 232448, "does not fit");
};

template <int D_HEAD, int G, int DT>
__global__ void __launch_bounds__(PdCfg<D_HEAD>::THREADS, 1) kvd_prefill_attn_dual_kernel(const __grid_constant__ PrefillParams P) {
  using Cfg = PdCfg<D_HEAD>;
  constexpr int TOK = PT_ROWS / G;
  constexpr int SLOTS = Cfg::SLOTS, SLOTS_K = Cfg::SLOTS_K, SLOTS_V = Cfg::SLOTS_V;
  extern __shared__ uint8_t pt_smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort_i, s_lo[2], s_hi[2];  // first and last key position a tile needs
  volatile int *s_abort = &s_abort_i;
  const uint32_t q_smem = (smem_u32(pt_smem_raw) + 1023u) & ~1023u;  // the swizzle is a function of the address
  const uint32_t ring = q_smem + 2 * Cfg::Q_BYTES, ring_v = ring + SLOTS_K * Cfg::TILE_BYTES;
  const uint32_t bar_base = ring + SLOTS * Cfg::TILE_BYTES;
  auto bar_full = [&](int v, int s) { return bar_base + 8u * (v * SLOTS_K + s); };           // a block has landed
  auto bar_empty = [&](int v, int s) { return bar_base + 8u * (SLOTS + v * SLOTS_K + s); };  // both tiles' products with it are done
  auto bar_s_full = [&](int t, int b) { return bar_base + 8u * (2 * SLOTS + 2 * t + b); };       // scores of a block
  auto bar_p_ready = [&](int t, int b) { return bar_base + 8u * (2 * SLOTS + 4 + 2 * t + b); };  // weights in place
  auto bar_pv_done = [&](int t) { return bar_base + 8u * (2 * SLOTS + 8 + t); };                 // O += P V finished
  auto bar_o_full = [&](int t) { return bar_base + 8u * (2 * SLOTS + 10 + t); };
  auto bar_q_ready = [&](int t) { return bar_base + 8u * (2 * SLOTS + 12 + t); };
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  // start order as above: late tokens first, for every pair of tiles all KV heads before the next shorter one
  const int n_pairs = static_cast<int>(gridDim.x) / P.n_kv;
  const int kvh = static_cast<int>(blockIdx.x) % P.n_kv;
  const int cta_tok0 = (n_pairs - 1 - static_cast<int>(blockIdx.x) / P.n_kv) * 2 * TOK;
  const unsigned long long tmo = P.timeout_ns;

  if (tid == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(bar_full(0, s), Cfg::LOADERS / 32);  // one arrival per loader warp
      mbar_init(bar_empty(0, s), 2);                 // the commits of both tiles
    }
    for (int t = 0; t < 2; ++t) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(bar_s_full(t, b), 1);
        mbar_init(bar_p_ready(t, b), 4);  // one arrival per softmax warp of the tile
      }
      mbar_init(bar_pv_done(t), 1);
      mbar_init(bar_o_full(t), 1);
      mbar_init(bar_q_ready(t), 4);
    }
    fence_mbar_init();
    s_abort_i = 0;
    for (int t = 0; t < 2; ++t) {
      s_lo[t] = INT_MAX;
      s_hi[t] = -1;
    }
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&s_tmem), Cfg::COLS);
    tmem_relinquish();
  }
  __syncthreads();
  early_start_point();
  // ---- key positions a tile needs: from the smallest first-visible to the largest last-visible of its tokens
  if (tid < 2 * TOK && cta_tok0 + tid < P.n_rows) {
    const int qp = P.q_pos[cta_tok0 + tid];
    int lo = first_visible(qp, P.window);
    lo = lo < P.seg_lo ? P.seg_lo : lo;
    const int hi = qp < P.seg_hi ? qp : P.seg_hi;
    if (hi >= lo) {
      atomicMin(&s_lo[tid / TOK], lo);
      atomicMax(&s_hi[tid / TOK], hi);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = s_tmem;
  // The blocks the CTA loads, and the ones of these that tile t takes: its own range and no more.  In a block only the
  // other tile sees, an infinity or a NaN in V would reach this tile's rows as a weight of 0 times it.
  const int hi_all = s_hi[0] > s_hi[1] ? s_hi[0] : s_hi[1], lo_all = s_lo[0] < s_lo[1] ? s_lo[0] : s_lo[1];
  const int blk0 = hi_all >= 0 ? lo_all / PT_KEYS : 0;
  const int n_blk = hi_all >= 0 ? hi_all / PT_KEYS - blk0 + 1 : 0;
  auto tile_skip = [&](int t) { return s_hi[t] >= 0 ? s_lo[t] / PT_KEYS - blk0 : 0; };                        // blocks before its first
  auto tile_blocks = [&](int t) { return s_hi[t] >= 0 ? s_hi[t] / PT_KEYS - s_lo[t] / PT_KEYS + 1 : 0; };

  if (warp < 8) {
    // ------------------------------------------------------------------ softmax and epilogue: thread = MMA row of tile t
    const int t = warp >> 2, q4 = warp & 3;
    const int row = q4 * 32 + lane;
    const int tok = cta_tok0 + t * TOK + row / G, g = row % G;
    const bool valid = row / G < TOK && tok < P.n_rows;
    const int qp = valid ? P.q_pos[tok] : -1;
    const int lo = first_visible(qp, P.window);
    const int first_blk = blk0 + tile_skip(t), n = tile_blocks(t);
    const uint32_t lane_field = static_cast<uint32_t>(q4 * 32) << 16;
    const uint32_t o_col = tmem_base + lane_field + t * D_HEAD;
    const size_t row_off = (static_cast<size_t>(valid ? tok : 0) * P.n_q + kvh * G + (valid ? g : 0)) * D_HEAD;
    if (n > 0) {
      // the query row into shared memory, K-major with the 128-byte swizzle (zeros for padding rows)
      const uint4 *qsrc = reinterpret_cast<const uint4 *>(P.q + row_off);
      const uint32_t qdst = q_smem + t * Cfg::Q_BYTES + row * 128;
#pragma unroll
      for (int c = 0; c < D_HEAD / 8; ++c) {
        const uint4 w = valid ? qsrc[c] : make_uint4(0u, 0u, 0u, 0u);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(qdst + (c >> 3) * Cfg::SLAB_Q + (((c & 7) ^ (row & 7)) << 4)), "r"(w.x), "r"(w.y),
                     "r"(w.z), "r"(w.w)
                     : "memory");
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_q_ready(t));
    }
    // the two parts of the row sum (blocks of this and of the other parity), each with the reference it had last
    float m_run = -CUDART_INF_F, m_own = -CUDART_INF_F, m_other = -CUDART_INF_F;
    uint64_t l2[2] = {0ull, 0ull}, l2_other[2] = {0ull, 0ull};
    bool ok = true;
    const uint64_t c2 = pack2(P.scale_log2e, P.scale_log2e);
    PtWhole whole_block(valid, lo, qp);
    for (int j = 0; j < n; ++j) {
      const int buf = j & 1;
      if (!polite_warp_wait(bar_s_full(t, buf), (j >> 1) & 1, s_abort, tmo, lane)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t s_col = tmem_base + lane_field + Cfg::COL_S + (2 * t + buf) * PT_KEYS;
      uint32_t s0[32], s1[32];
      tmem_ld_x32(s_col, s0);
      tmem_ld_x32(s_col + 32, s1);
      const bool whole = whole_block(P, (first_blk + j) * PT_KEYS);  // (warp-uniform)
      unsigned long long vis = ~0ull;
      if (!whole) vis = pt_visible(P, (first_blk + j) * PT_KEYS, lo, qp);
      tmem_wait_ld();
      const float bm = pt_mask_max(s0, s1, whole, vis) * P.scale_log2e;  // log2 units (scale > 0)
      // the lazy reference of the kernel above
      const float m_prev = m_run;
      m_run = m_prev == -CUDART_INF_F ? bm : (bm > m_prev + PT_TAU ? bm : m_prev);
      const float m_use = m_run == -CUDART_INF_F ? 0.f : m_run;
      const float alpha = m_prev == -CUDART_INF_F ? 1.0f : ex2_approx(m_prev - m_use);
      const float alpha_own = m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use);
      m_own = m_run;
      uint32_t w[32];
      const uint64_t al2 = pack2(alpha_own, alpha_own);
      l2[0] = fmul2(l2[0], al2);
      l2[1] = fmul2(l2[1], al2);
      pt_weights<DT>(s0, s1, c2, pack2(-m_use, -m_use), l2, w);
      tmem_st_x32(s_col, w);  // over the scores, which are in registers
      if (__any_sync(0xffffffffu, alpha != 1.0f)) {
        // O holds the blocks before j (j >= 1 here: a maximum exists); the last of those products must have finished
        if (!polite_warp_wait(bar_pv_done(t), (j - 1) & 1, s_abort, tmo, lane)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
          break;
        }
        tc_fence_after();
        pt_rescale<D_HEAD>(o_col, alpha);
      } else {
        tmem_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p_ready(t, buf));
      // the next block belongs to the other part
      const float mt = m_own;
      m_own = m_other;
      m_other = mt;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint64_t lt = l2[i];
        l2[i] = l2_other[i];
        l2_other[i] = lt;
      }
    }
    // ---- the row sum: both parts referred to the final maximum (a sum of two: the order does not matter)
    float l_run = 0.f;
    if (ok && n > 0) {
      const float m_use = m_run == -CUDART_INF_F ? 0.f : m_run;
      l_run = pt_row_sum(l2, m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use)) +
              pt_row_sum(l2_other, m_other == -CUDART_INF_F ? 1.0f : ex2_approx(m_other - m_use));
      if (!polite_warp_wait(bar_o_full(t), 0, s_abort, tmo, lane)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
      }
    }
    // ---- normalise and store (a token without a visible key yields zeros)
    if (ok) {
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
      uint4 *dst = reinterpret_cast<uint4 *>(P.out + row_off);
#pragma unroll 1
      for (int c = 0; c < D_HEAD / 32; ++c) {
        uint32_t r[32];
        if (n > 0) {
          tmem_ld_x32(o_col + c * 32, r);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
        }
        uint32_t o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = pack_out<DT>(__uint_as_float(r[2 * i]) * inv, __uint_as_float(r[2 * i + 1]) * inv);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 4; ++i) dst[c * 4 + i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
        }
      }
    }
  } else if (warp < 10) {
    // ------------------------------------------------------------------ both products of tile t (one thread)
    constexpr uint32_t IDESC_BASE = (DT == 0 ? umma_idesc_bf16_f32(PT_ROWS, 8) : umma_idesc_f16_f32(PT_ROWS, 8)) & ~(1u << 17);
    constexpr uint32_t IDESC_S = IDESC_BASE | (static_cast<uint32_t>(PT_KEYS >> 3) << 17);              // N = 64 keys, B K-major
    constexpr uint32_t IDESC_O = IDESC_BASE | (static_cast<uint32_t>(D_HEAD >> 3) << 17) | (1u << 16);  // N = d_head, B MN-major
    const int t = warp - 8;
    if (n_blk > 0 && elect_one()) {
      const int skip = tile_skip(t), n = tile_blocks(t);
      // blocks that only the other tile takes: released when they have landed (not earlier: the next phase of the
      // slot's barrier must not get this tile's arrival before the other tile's of this phase)
      auto pass = [&](int from, int to) -> bool {
        for (int b = from; b < to; ++b)
          for (int v = 0; v < 2; ++v) {
            const int slots = v ? SLOTS_V : SLOTS_K, slot = b % slots;
            if (!polite_wait<false>(bar_full(v, slot), (b / slots) & 1, s_abort, tmo)) return false;
            mbar_arrive(bar_empty(v, slot));
          }
        return true;
      };
      bool ok = pass(0, skip);
      if (ok && n > 0) ok = polite_wait<false>(bar_q_ready(t), 0, s_abort, tmo);
      auto scores = [&](int j) -> bool {
        const int slot = (skip + j) % SLOTS_K;
        if (!polite_wait<false>(bar_full(0, slot), ((skip + j) / SLOTS_K) & 1, s_abort, tmo)) return false;
        tc_fence_after();
        const uint32_t d = tmem_base + Cfg::COL_S + (2 * t + (j & 1)) * PT_KEYS;
        const uint64_t qdesc0 = umma_smem_desc_sw128(q_smem + t * Cfg::Q_BYTES), kdesc0 = umma_smem_desc_sw128(ring + slot * Cfg::TILE_BYTES);
#pragma unroll
        for (int ks = 0; ks < D_HEAD / 16; ++ks)
          umma_bf16(d, qdesc0 + (((ks >> 2) * Cfg::SLAB_Q + (ks & 3) * 32) >> 4), kdesc0 + (((ks >> 2) * Cfg::SLAB_K + (ks & 3) * 32) >> 4), IDESC_S,
                    ks > 0 ? 1u : 0u);
        umma_commit(bar_empty(0, slot));
        umma_commit(bar_s_full(t, j & 1));
        return true;
      };
      if (ok && n > 0) ok = scores(0);
      if (ok && n > 1) ok = scores(1);
      for (int j = 0; ok && j < n; ++j) {
        const int slot = (skip + j) % SLOTS_V;
        // the weights are in place (and O has been rescaled where a reference maximum moved), the V block has landed
        if (!polite_wait<false>(bar_p_ready(t, j & 1), (j >> 1) & 1, s_abort, tmo) ||
            !polite_wait<false>(bar_full(1, slot), ((skip + j) / SLOTS_V) & 1, s_abort, tmo)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t vdesc0 = umma_smem_desc_sw128_mn(ring_v + slot * Cfg::TILE_BYTES, Cfg::SLAB_V);
        const uint32_t p_col = tmem_base + Cfg::COL_S + (2 * t + (j & 1)) * PT_KEYS;
#pragma unroll
        for (int ks = 0; ks < PT_KEYS / 16; ++ks)
          umma_f16_ts(tmem_base + t * D_HEAD, p_col + ks * 8, vdesc0 + ((ks * 16 * 128) >> 4), IDESC_O, (j > 0 || ks > 0) ? 1u : 0u);
        umma_commit(bar_empty(1, slot));
        umma_commit(bar_pv_done(t));
        // (the next scores of this buffer are not urgent: they wait for the product that reads the weights in it)
        if (j + 2 < n) ok = polite_wait<false>(bar_pv_done(t), j & 1, s_abort, tmo) && scores(j + 2);
      }
      if (ok) umma_commit(bar_o_full(t));
      if (ok) ok = pass(skip + n, n_blk);
      if (!ok) raise(P.status, STATUS_TIMEOUT, s_abort);
    }
  } else {
    auto arrive = [&](uint32_t bar) { mbar_arrive(bar); };
    pt_load_blocks<Cfg, D_HEAD>(P, ring, ring_v, bar_base, SLOTS, blk0, n_blk, kvh, 0, tid - 10 * 32, arrive, s_abort, tmo);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::COLS);
  }
}

// ------------------------------------------------------------------------------------------------
// One row tile on two SMs (d_head 128 and 256), for launches whose tiles leave half of the GPU idle: then a tile's walk
// over its keys is the launch's length.  A cluster of two CTAs shares the tile: of every four key blocks CTA 0 takes the
// scores and weights of the first two and CTA 1 those of the last two (K blocks are loaded by the CTA that scores them),
// the weights go to both, and each CTA sums P V of every block over its half of the channels.
// The bits are those of the kernels above: the same blocks in the same order, an output element still is one
// accumulator, the reference maximum still passes from block to block, and a part of the row sum (even, odd blocks) still
// is one chain of additions, handed from one CTA to the other.
//   TMEM  = [ O : d_head / 2 columns | S_0, S_1 | Q ]
//   warps = 0-7 softmax (group = block parity), 8 issues S of this CTA's blocks, 9 P V of all blocks, 10 and 11 load K and
//           V, 12-15 rescale O where a reference maximum moved (the softmax warps of the other CTA cannot do it here).
//   P     = four blocks of weights in shared memory; the CTA that made a block copies it into the other's
//           (4 KB per warp, counted on the barrier the product waits on).
//   m     = a block's reference maxima go to both CTAs (eight slots); the row sums' chains go to the other CTA only.
// Across the pair everything travels with its own byte count on the receiver's barrier (st.async, bulk copies): nobody
// waits for a store to be performed.  A barrier that counts bytes is armed by one thread of the receiver.
// Bound by a softmax warp's chain of latencies: about 3600 clocks for one block of four (scores 450, maximum 280, weights
// 800 to 1000, six hand-overs).  Gemma-3-4B layer, 837 tokens on 7013, call alone: 123 -> 72.5 us (56 tiles on 112 SMs
// instead of 56).  Clock counts by phase led there: K and V gathered by cp.async 136 us, TMA by one warp 100, by one warp
// each 89, cheaper waits 81, and the early start.
template <int D_HEAD>
struct PsCfg {
  static constexpr int THREADS = 512, V_COLS = D_HEAD / 2;
  static constexpr int SLAB_K = PT_KEYS * 128, SLAB_V = PT_KEYS * 128;
  static constexpr int TILE_K = PT_KEYS * D_HEAD * 2, TILE_V = PT_KEYS * V_COLS * 2;
  static constexpr int SLOTS_K = D_HEAD == 256 ? 3 : 5, SLOTS_V = D_HEAD == 256 ? 3 : 6, SLOTS = SLOTS_K + SLOTS_V;
  static constexpr int P_SLOTS = 4, P_BYTES = PT_ROWS * PT_KEYS * 2;
  static constexpr int M_SLOTS = 8;
  static constexpr int COL_O = 0, COL_S = D_HEAD / 2, COL_Q = COL_S + 2 * PT_KEYS;
  static constexpr int COLS = D_HEAD == 256 ? 512 : 256;
  // full, empty | s_full[2] s_free[2] q_ready o_full | p_ready[4] | pv_done[8] scaled[8] | m[8][4] | chain[2][4] sum[2][4]
  // (Eight of what a block's maxima run ahead of: they may be seven blocks ahead of the products, and a barrier's phase can
  // only be told from the one before it.)
  static constexpr int N_BARS = 2 * SLOTS + 6 + 4 + 16 + 32 + 16;
  static constexpr int RINGS = SLOTS_K * TILE_K + SLOTS_V * TILE_V;
  static constexpr int SMEM_BYTES = 1024 + RINGS + P_SLOTS * P_BYTES + N_BARS * 8;
  static_assert(COL_Q + D_HEAD / 2 <= COLS && SMEM_BYTES + 9 * 1024 + 512 <= 232448, "does not fit");
};

// Maps of the segments' K and V rows (segment s: 2 s and 2 s + 1), boxes of 64 channels x 64 keys.
struct PsMaps {
  CUtensorMap map[2 * KVD_MAX_SEGMENTS];
};

// A loader warp: n blocks of K (IS_V false) or V of the walk, the t-th of them block_of(t), into the ring of `slots` tiles
// at `ring`; of V the channels from v_col on.  A block inside one segment is fetched by TMA: the rings are short, and what
// counts is that a free slot's bytes are under way at once (with 16-byte cp.async from two warps the scores waited for K
// blocks 83 % of the time, with one warp loading both by TMA still 70 %).  A block across segments, or with positions
// nobody holds, is gathered.
template <class Cfg, int D_HEAD, bool IS_V, class BlockOf>
__device__ __forceinline__ void ps_load_blocks(const PrefillParams &P, const PsMaps &maps, uint32_t ring, uint32_t bar_base, int blk0, int n, int kvh,
                                               int v_col, const BlockOf &block_of, int lane, volatile int *s_abort, unsigned long long tmo) {
  constexpr int slots = IS_V ? Cfg::SLOTS_V : Cfg::SLOTS_K, tile = IS_V ? Cfg::TILE_V : Cfg::TILE_K, cols = IS_V ? Cfg::V_COLS : D_HEAD;
  const int col0 = kvh * D_HEAD + (IS_V ? v_col : 0);
  bool ok = true;
  for (int t = 0; t < n; ++t) {
    const int slot = t % slots;
    const uint32_t full = bar_base + 8u * ((IS_V ? Cfg::SLOTS_K : 0) + slot), empty = full + 8u * Cfg::SLOTS;
    if (t >= slots && !polite_warp_wait(empty, ((t / slots) - 1) & 1, s_abort, tmo, lane)) {
      ok = false;
      break;
    }
    const uint32_t dst = ring + slot * tile;
    const int pos0 = (blk0 + block_of(t)) * PT_KEYS;
    int whole = -1;
#pragma unroll
    for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg)
      if (segment_holds(P.first[sg], P.len[sg], pos0, PT_KEYS)) whole = sg;
    if (whole >= 0) {
      if (elect_one()) {
        mbar_arrive_expect_tx(full, tile);
        const CUtensorMap *map = &maps.map[2 * whole + (IS_V ? 1 : 0)];
#pragma unroll
        for (int c = 0; c < cols; c += 64) tma_load_2d(dst + (c >> 6) * (PT_KEYS * 128), map, full, col0 + c, pos0 - P.first[whole]);
      }
      __syncwarp();
      continue;
    }
#pragma unroll 1
    for (int i = lane; i < PT_KEYS * (cols / 8); i += 32) {  // 16-byte pieces
      const int r = i / (cols / 8), c = i % (cols / 8), pos = pos0 + r;
      const __nv_bfloat16 *src = P.q;
      bool have = false;
#pragma unroll
      for (int sg = 0; sg < KVD_MAX_SEGMENTS; ++sg) {
        const int rr = pos - P.first[sg];
        if (rr >= 0 && rr < P.len[sg]) {
          src = (IS_V ? P.v[sg] : P.k[sg]) + static_cast<size_t>(rr) * P.stride[sg] + col0 + c * 8;
          have = true;
        }
      }
      cp_async16(dst + (c >> 3) * (PT_KEYS * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, have);
    }
    cp_async_wait_all();
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(full);
  }
  if (!ok) {
    raise(P.status, STATUS_TIMEOUT, s_abort);
    // copies may still be in flight: a bounded time that exceeds any load's latency by orders of magnitude
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
  }
}

template <int D_HEAD, int G, int DT>
__global__ void __launch_bounds__(PsCfg<D_HEAD>::THREADS, 1)
    kvd_prefill_attn_split_kernel(const __grid_constant__ PrefillParams P, const __grid_constant__ PsMaps maps) {
  using Cfg = PsCfg<D_HEAD>;
  constexpr int TOK = PT_ROWS / G, HALF = D_HEAD / 2;
  constexpr int SLOTS = Cfg::SLOTS, SLOTS_K = Cfg::SLOTS_K, SLOTS_V = Cfg::SLOTS_V;
  extern __shared__ uint8_t pt_smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort_i, s_lo, s_hi;
  __shared__ float s_m[Cfg::M_SLOTS][PT_ROWS];                // reference maximum after a block
  __shared__ __align__(16) uint4 s_chain[2][PT_ROWS];         // a part of the row sum after the other CTA's block
  __shared__ float s_sum[2][PT_ROWS];                         // the parts, referred to the last maximum
  volatile int *s_abort = &s_abort_i;
  const uint32_t ring = (smem_u32(pt_smem_raw) + 1023u) & ~1023u, ring_v = ring + SLOTS_K * Cfg::TILE_K;
  const uint32_t p_smem = ring + Cfg::RINGS, bar_base = p_smem + Cfg::P_SLOTS * Cfg::P_BYTES;
  auto bar = [&](int i) { return bar_base + 8u * static_cast<uint32_t>(i); };
  auto bar_full = [&](int v, int s) { return bar(v * SLOTS_K + s); };
  auto bar_empty = [&](int v, int s) { return bar(SLOTS + v * SLOTS_K + s); };
  constexpr int B0 = 2 * SLOTS;
  auto bar_s_full = [&](int b) { return bar(B0 + b); };
  auto bar_s_free = [&](int b) { return bar(B0 + 2 + b); };
  const uint32_t bar_q_ready = bar(B0 + 4), bar_o_full = bar(B0 + 5);
  auto bar_p_ready = [&](int j) { return bar(B0 + 6 + (j & 3)); };
  auto bar_pv_done = [&](int j) { return bar(B0 + 10 + (j & 7)); };  // both CTAs' products with the block
  auto bar_scaled = [&](int j) { return bar(B0 + 18 + (j & 7)); };   // O is ready for the block
  auto bar_m = [&](int j, int q) { return bar(B0 + 26 + (j & 7) * 4 + q); };
  auto bar_chain = [&](int g, int q) { return bar(B0 + 58 + g * 4 + q); };
  auto bar_sum = [&](int g, int q) { return bar(B0 + 66 + g * 4 + q); };

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const uint32_t other = static_cast<uint32_t>(rank ^ 1);
  // start order as above: late tokens first, for every tile all KV heads before the next shorter one
  const int n_tiles = static_cast<int>(gridDim.x) / (2 * P.n_kv), slot_id = static_cast<int>(blockIdx.x) / 2;
  const int kvh = slot_id % P.n_kv;
  const int tok0 = (n_tiles - 1 - slot_id / P.n_kv) * TOK;
  const unsigned long long tmo = P.timeout_ns;
  auto owner = [](int j) { return (j >> 1) & 1; };  // the CTA that scores block j

  if (tid == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(bar_full(0, s), 1);   // the loader's lane, and the block's bytes where TMA brings them
      mbar_init(bar_empty(0, s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_s_full(b), 1);
      mbar_init(bar_s_free(b), 4);
    }
    mbar_init(bar_q_ready, 8);
    mbar_init(bar_o_full, 1);
    for (int s = 0; s < 4; ++s) {
      mbar_init(bar_p_ready(s), owner(s) == rank ? 4 : 1);  // its four warps here, or the arming thread and 16 KB
    }
    for (int s = 0; s < 8; ++s) {
      mbar_init(bar_pv_done(s), 2);
      mbar_init(bar_scaled(s), 4);
    }
    for (int i = 0; i < 32 + 16; ++i) mbar_init(bar(B0 + 26 + i), 1);
    fence_mbar_init();
    s_abort_i = 0;
    s_lo = INT_MAX;
    s_hi = -1;
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&s_tmem), Cfg::COLS);
    tmem_relinquish();
  }
  __syncthreads();
  early_start_point();
  if (tid < TOK && tok0 + tid < P.n_rows) {
    const int qp = P.q_pos[tok0 + tid];
    int lo = first_visible(qp, P.window);
    lo = lo < P.seg_lo ? P.seg_lo : lo;
    const int hi = qp < P.seg_hi ? qp : P.seg_hi;
    if (hi >= lo) {
      atomicMin(&s_lo, lo);
      atomicMax(&s_hi, hi);
    }
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = s_tmem;
  const int blk0 = s_hi >= 0 ? s_lo / PT_KEYS : 0;
  const int n_blk = s_hi >= 0 ? s_hi / PT_KEYS - blk0 + 1 : 0;
  const int last4 = (n_blk & 3) - 2 * rank, n_own = (n_blk >> 2) * 2 + (last4 < 0 ? 0 : last4 > 2 ? 2 : last4);  // blocks this CTA scores
  auto own_block = [&](int t) { return 4 * (t >> 1) + 2 * rank + (t & 1); };
  // waits on what the other CTA completes, alone or in turn with this one
  auto peer_wait = [&](uint32_t b, uint32_t parity) -> bool { return polite_warp_wait<true>(b, parity, s_abort, tmo, lane); };
  auto m_at = [&](int j, int row) { return smem_u32(&s_m[j & 7][row]); };

  if (warp < 8) {
    // ------------------------------------------------------------------ softmax and epilogue: thread = MMA row
    const int wg = warp >> 2, q4 = warp & 3;
    const int row = q4 * 32 + lane;
    const int tok = tok0 + row / G, g = row % G;
    const bool valid = row / G < TOK && tok < P.n_rows;
    const int qp = valid ? P.q_pos[tok] : -1;
    const int lo = first_visible(qp, P.window);
    const uint32_t lane_field = static_cast<uint32_t>(q4 * 32) << 16;
    const size_t row_off = (static_cast<size_t>(valid ? tok : 0) * P.n_q + kvh * G + (valid ? g : 0)) * D_HEAD;
    if (n_blk > 0) {
      const uint4 *qsrc = reinterpret_cast<const uint4 *>(P.q + row_off);
#pragma unroll 1
      for (int c = wg; c < D_HEAD / 64; c += 2) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 w = valid ? qsrc[c * 8 + i] : make_uint4(0u, 0u, 0u, 0u);
          r[4 * i] = w.x;
          r[4 * i + 1] = w.y;
          r[4 * i + 2] = w.z;
          r[4 * i + 3] = w.w;
        }
        tmem_st_x32(tmem_base + lane_field + Cfg::COL_Q + c * 32, r);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_q_ready);
    }
    const uint32_t chain_bar = bar_chain(wg, q4);
    if (lane == 0) mbar_arrive_expect_tx(chain_bar, 512);
    uint32_t chain_ph = 0;
    float m_own = -CUDART_INF_F;
    uint64_t l2[2] = {0ull, 0ull};
    bool ok = true, have_part = false;  // have_part: this group took the last block of its parity
    const uint64_t c2 = pack2(P.scale_log2e, P.scale_log2e), one2 = pack2(1.0f, 1.0f);
    PtWhole whole_block(valid, lo, qp);
    for (int j = 2 * rank + wg; j < n_blk; j += 4) {
      if (!polite_warp_wait(bar_s_full(wg), (j >> 2) & 1, s_abort, tmo, lane)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t s_col = tmem_base + lane_field + Cfg::COL_S + wg * PT_KEYS;
      uint32_t s0[32], s1[32];
      tmem_ld_x32(s_col, s0);
      tmem_ld_x32(s_col + 32, s1);
      const bool whole = whole_block(P, (blk0 + j) * PT_KEYS);  // (warp-uniform)
      unsigned long long vis = ~0ull;
      if (!whole) vis = pt_visible(P, (blk0 + j) * PT_KEYS, lo, qp);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_s_free(wg));
      const float bm = pt_mask_max(s0, s1, whole, vis) * P.scale_log2e;
      float m_prev = -CUDART_INF_F;
      if (j > 0) {
        if (!peer_wait(bar_m(j - 1, q4), ((j - 1) >> 3) & 1)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
          break;
        }
        m_prev = s_m[(j - 1) & 7][row];
      }
      const float m_new = m_prev == -CUDART_INF_F ? bm : (bm > m_prev + PT_TAU ? bm : m_prev);
      s_m[j & 7][row] = m_new;
      st_async_f32(map_to_cta(m_at(j, row), other), map_to_cta(bar_m(j, q4), other), m_new);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_m(j, q4));
      const float m_use = m_new == -CUDART_INF_F ? 0.f : m_new;
      // both CTAs' products with the weights that were in this slot have finished
      if (j >= 4 && !peer_wait(bar_pv_done(j - 4), ((j - 4) >> 3) & 1)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
        break;
      }
      const uint64_t nm2 = pack2(-m_use, -m_use);
      const uint32_t p_slot = p_smem + (j & 3) * Cfg::P_BYTES, prow = p_slot + row * 128;
      auto weights = [&](uint32_t (&s)[32], int chunk0) {  // in fp32 over the scores, rounded into the slot
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k = 8 * c + 2 * i;
            float e0, e1;
            unpack2(ffma2(pack2(__uint_as_float(s[k]), __uint_as_float(s[k + 1])), c2, nm2), e0, e1);
            const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);
            w[i] = pack_out<DT>(p0, p1);
            s[k] = __float_as_uint(p0);
            s[k + 1] = __float_as_uint(p1);
          }
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(prow + (((chunk0 + c) ^ (row & 7)) << 4)), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                       "r"(w[3])
                       : "memory");
        }
      };
      weights(s0, 0);
      weights(s1, 4);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_p_ready(j));
        const uint32_t piece = p_slot + q4 * 4096;
        bulk_copy_to_cta(map_to_cta(piece, other), piece, 4096, map_to_cta(bar_p_ready(j), other));
      }
      // the row sum's part: the chain of block j - 2, which the other CTA took, and its reference
      if (j >= 2) {
        const uint32_t m_bar = bar_m(j - 2, q4), m_ph = ((j - 2) >> 3) & 1;
        const bool both = mbar_try_wait_cluster(chain_bar, chain_ph) && mbar_try_wait_cluster(m_bar, m_ph);
        if (!__all_sync(0xffffffffu, both) && (!peer_wait(chain_bar, chain_ph) || !peer_wait(m_bar, m_ph))) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          ok = false;
          break;
        }
        chain_ph ^= 1u;
        const uint4 c = s_chain[wg][row];
        l2[0] = pack2(__uint_as_float(c.x), __uint_as_float(c.y));
        l2[1] = pack2(__uint_as_float(c.z), __uint_as_float(c.w));
        m_own = s_m[(j - 2) & 7][row];
        __syncwarp();
        if (lane == 0) mbar_arrive_expect_tx(chain_bar, 512);
      }
      const float alpha_own = m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use);
      m_own = m_new;
      const uint64_t al2 = pack2(alpha_own, alpha_own);
      l2[0] = fmul2(l2[0], al2);
      l2[1] = fmul2(l2[1], al2);
#pragma unroll
      for (int k = 0; k < 32; k += 2) l2[(k >> 1) & 1] = ffma2(pack2(__uint_as_float(s0[k]), __uint_as_float(s0[k + 1])), one2, l2[(k >> 1) & 1]);
#pragma unroll
      for (int k = 0; k < 32; k += 2) l2[(k >> 1) & 1] = ffma2(pack2(__uint_as_float(s1[k]), __uint_as_float(s1[k + 1])), one2, l2[(k >> 1) & 1]);
      have_part = j + 2 >= n_blk;
      if (!have_part) {
        float a0, a1, a2, a3;
        unpack2(l2[0], a0, a1);
        unpack2(l2[1], a2, a3);
        st_async_v4(map_to_cta(smem_u32(&s_chain[wg][row]), other), map_to_cta(chain_bar, other), __float_as_uint(a0), __float_as_uint(a1),
                    __float_as_uint(a2), __float_as_uint(a3));
      }
    }
    // ---- the row sum: both parts referred to the final maximum, added in group order
    float l_run = 0.f;
    if (ok && n_blk > 0) {
      const int last = n_blk - 1;
      if (!peer_wait(bar_m(last, q4), (last >> 3) & 1)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
      }
      if (ok && wg <= last) {
        if (have_part) {
          const float m_fin = s_m[last & 7][row], m_use = m_fin == -CUDART_INF_F ? 0.f : m_fin;
          const float part = pt_row_sum(l2, m_own == -CUDART_INF_F ? 1.0f : ex2_approx(m_own - m_use));
          s_sum[wg][row] = part;
          st_async_f32(map_to_cta(smem_u32(&s_sum[wg][row]), other), map_to_cta(bar_sum(wg, q4), other), part);
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_sum(wg, q4));
        } else if (lane == 0) {
          mbar_arrive_expect_tx(bar_sum(wg, q4), 128);
        }
      }
      if (ok && (!peer_wait(bar_sum(0, q4), 0) || (last > 0 && !peer_wait(bar_sum(1, q4), 0)))) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        ok = false;
      }
      if (ok) l_run = s_sum[0][row] + (last > 0 ? s_sum[1][row] : 0.f);
    }
    // ---- normalise and store this CTA's channels, each group its pieces of 32
    if (ok && n_blk > 0 && !polite_warp_wait(bar_o_full, 0, s_abort, tmo, lane)) {
      raise(P.status, STATUS_TIMEOUT, s_abort);
      ok = false;
    }
    if (ok) {
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
      uint4 *dst = reinterpret_cast<uint4 *>(P.out + row_off + rank * HALF);
#pragma unroll 1
      for (int c = wg; c < HALF / 32; c += 2) {
        uint32_t r[32];
        if (n_blk > 0) {
          tmem_ld_x32(tmem_base + lane_field + Cfg::COL_O + c * 32, r);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
        }
        uint32_t o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = pack_out<DT>(__uint_as_float(r[2 * i]) * inv, __uint_as_float(r[2 * i + 1]) * inv);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 4; ++i) dst[c * 4 + i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
        }
      }
    } else {
      // copies of this warp may still be on their way into the other CTA (which stays until the barrier below)
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
  } else if (warp == 8 || warp == 9) {
    // ------------------------------------------------------------------ MMA issue (one thread per product)
    constexpr uint32_t IDESC_BASE = (DT == 0 ? umma_idesc_bf16_f32(PT_ROWS, 8) : umma_idesc_f16_f32(PT_ROWS, 8)) & ~(1u << 17);
    constexpr uint32_t IDESC_S = IDESC_BASE | (static_cast<uint32_t>(PT_KEYS >> 3) << 17);            // N = 64 keys, B K-major
    constexpr uint32_t IDESC_O = IDESC_BASE | (static_cast<uint32_t>(HALF >> 3) << 17) | (1u << 16);  // N = d_head / 2, B MN-major
    if (warp == 8 && n_own > 0 && elect_one()) {
      bool ok = polite_wait<false>(bar_q_ready, 0, s_abort, tmo);
      tc_fence_after();
      for (int t = 0; ok && t < n_own; ++t) {
        const int slot = t % SLOTS_K;
        if (!polite_wait<false>(bar_full(0, slot), (t / SLOTS_K) & 1, s_abort, tmo) ||
            (t >= 2 && !polite_wait<false>(bar_s_free(t & 1), ((t - 2) >> 1) & 1, s_abort, tmo))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem_base + Cfg::COL_S + (t & 1) * PT_KEYS;
        const uint64_t desc0 = umma_smem_desc_sw128(ring + slot * Cfg::TILE_K);
#pragma unroll
        for (int ks = 0; ks < D_HEAD / 16; ++ks)
          umma_f16_ts(d, tmem_base + Cfg::COL_Q + ks * 8, desc0 + (((ks >> 2) * Cfg::SLAB_K + (ks & 3) * 32) >> 4), IDESC_S, ks > 0 ? 1u : 0u);
        umma_commit(bar_empty(0, slot));
        umma_commit(bar_s_full(t & 1));
      }
      if (!ok) raise(P.status, STATUS_TIMEOUT, s_abort);
    } else if (warp == 9 && n_blk > 0 && elect_one()) {
      bool ok = true;
      for (int s = 0; s < 4; ++s)
        if (owner(s) != rank) mbar_arrive_expect_tx(bar_p_ready(s), Cfg::P_BYTES);
      for (int j = 0; j < n_blk; ++j) {
        const int slot = j % SLOTS_V;
        if (!polite_wait<false>(bar_scaled(j), (j >> 3) & 1, s_abort, tmo) || !polite_wait<true>(bar_p_ready(j), (j >> 2) & 1, s_abort, tmo) ||
            !polite_wait<false>(bar_full(1, slot), (j / SLOTS_V) & 1, s_abort, tmo)) {
          ok = false;
          break;
        }
        if (owner(j) != rank) mbar_arrive_expect_tx(bar_p_ready(j), Cfg::P_BYTES);  // for block j + 4
        tc_fence_after();
        const uint64_t desc0 = umma_smem_desc_sw128_mn(ring_v + slot * Cfg::TILE_V, Cfg::SLAB_V);
        const uint64_t pdesc0 = umma_smem_desc_sw128(p_smem + (j & 3) * Cfg::P_BYTES);
#pragma unroll
        for (int ks = 0; ks < PT_KEYS / 16; ++ks)
          umma_bf16(tmem_base + Cfg::COL_O, pdesc0 + ((ks * 32) >> 4), desc0 + ((ks * 16 * 128) >> 4), IDESC_O, (j > 0 || ks > 0) ? 1u : 0u);
        umma_commit(bar_empty(1, slot));
        umma_commit_mask(bar_pv_done(j), 3);
      }
      if (ok) umma_commit(bar_o_full);
      // the other CTA's last commits have arrived here before this one may leave
      for (int j = n_blk > 4 ? n_blk - 4 : 0; ok && j < n_blk; ++j) ok = polite_wait<true>(bar_pv_done(j), (j >> 3) & 1, s_abort, tmo);
      if (!ok) raise(P.status, STATUS_TIMEOUT, s_abort);
    }
  } else if (warp < 12) {
    if (warp == 10) ps_load_blocks<Cfg, D_HEAD, false>(P, maps, ring, bar_base, blk0, n_own, kvh, 0, own_block, lane, s_abort, tmo);
    else ps_load_blocks<Cfg, D_HEAD, true>(P, maps, ring_v, bar_base, blk0, n_blk, kvh, rank * HALF, [](int t) { return t; }, lane, s_abort, tmo);
  } else {
    // ------------------------------------------------------------------ O follows the reference maxima
    const int q4 = warp & 3, row = q4 * 32 + lane;
    const uint32_t o_col = tmem_base + (static_cast<uint32_t>(q4 * 32) << 16) + Cfg::COL_O;
    if (lane == 0)
      for (int j = 0; j < 8; ++j)
        if (owner(j) != rank) mbar_arrive_expect_tx(bar_m(j, q4), 128);
    float m_prev = -CUDART_INF_F;
    for (int j = 0; j < n_blk; ++j) {
      if (!peer_wait(bar_m(j, q4), (j >> 3) & 1)) {
        raise(P.status, STATUS_TIMEOUT, s_abort);
        break;
      }
      if (lane == 0 && owner(j) != rank) mbar_arrive_expect_tx(bar_m(j, q4), 128);  // for block j + 8
      const float m_new = s_m[j & 7][row], m_use = m_new == -CUDART_INF_F ? 0.f : m_new;
      const float alpha = m_prev == -CUDART_INF_F ? 1.0f : ex2_approx(m_prev - m_use);
      m_prev = m_new;
      if (__any_sync(0xffffffffu, alpha != 1.0f)) {
        if (!peer_wait(bar_pv_done(j - 1), ((j - 1) >> 3) & 1)) {
          raise(P.status, STATUS_TIMEOUT, s_abort);
          break;
        }
        tc_fence_after();
        pt_rescale<HALF>(o_col, alpha);
        tc_fence_before();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_scaled(j));
    }
  }
  // ---- nobody leaves while the other CTA can still write into its shared memory
  tc_fence_before();
  cluster_sync_all();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::COLS);
  }
}

template <typename... K, typename... A>
static kvd_status prefill_launch(kvd_ctx *ctx, void (*kern)(K...), unsigned grid, unsigned threads, size_t smem, unsigned cluster, cudaStream_t stream,
                                 const A &...args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = (serial_launch_mask() & 8) ? 0 : 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "launch prefill attention");
  ctx->launches += 1;
  return KVD_OK;
}

template <int D_HEAD, int G>
static kvd_status prefill_split_launch(kvd_ctx *ctx, const PrefillParams &P, cudaStream_t stream) {
  using Cfg = PsCfg<D_HEAD>;
  auto k0 = kvd_prefill_attn_split_kernel<D_HEAD, G, 0>;
  auto k1 = kvd_prefill_attn_split_kernel<D_HEAD, G, 1>;
  static bool configured[64] = {};
  if (!configured[ctx->device & 63]) {
    cudaError_t e = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute(prefill attention)");
    configured[ctx->device & 63] = true;
  }
  PsMaps maps;
  memset(&maps, 0, sizeof(maps));
  for (int i = 0; i < 2 * KVD_MAX_SEGMENTS; ++i) {
    const int sg = i / 2;
    if (P.len[sg] < PT_KEYS) continue;  // no block lies inside it
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(P.n_kv) * D_HEAD, static_cast<cuuint64_t>(P.len[sg])};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(P.stride[sg]) * 2};
    cuuint32_t box[2] = {64, PT_KEYS}, estr[2] = {1, 1};
    CUresult r = ctx->encode(&maps.map[i], ctx->dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                             const_cast<__nv_bfloat16 *>(i % 2 ? P.v[sg] : P.k[sg]), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      ctx->last_error = "cuTensorMapEncodeTiled (segments) failed: " + std::to_string(static_cast<int>(r));
      return KVD_ERR_CUDA;
    }
  }
  const int tok = PT_ROWS / G;
  return prefill_launch(ctx, ctx->dtype == 1 ? k1 : k0, 2 * ((P.n_rows + tok - 1) / tok) * P.n_kv, Cfg::THREADS, Cfg::SMEM_BYTES, 2, stream, P, maps);
}

template <int D_HEAD, int G>
static kvd_status prefill_dual_launch(kvd_ctx *ctx, const PrefillParams &P, cudaStream_t stream) {
  using Cfg = PdCfg<D_HEAD>;
  auto k0 = kvd_prefill_attn_dual_kernel<D_HEAD, G, 0>;
  auto k1 = kvd_prefill_attn_dual_kernel<D_HEAD, G, 1>;
  static bool configured[64] = {};
  if (!configured[ctx->device & 63]) {
    cudaError_t e = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute(prefill attention)");
    configured[ctx->device & 63] = true;
  }
  const int tok = 2 * (PT_ROWS / G);
  const unsigned grid = static_cast<unsigned>((P.n_rows + tok - 1) / tok * P.n_kv);
  return prefill_launch(ctx, ctx->dtype == 1 ? k1 : k0, grid, Cfg::THREADS, Cfg::SMEM_BYTES, 1, stream, P);
}

template <int D_HEAD, int G, bool PAIR>
static kvd_status prefill_tc_launch(kvd_ctx *ctx, const PrefillParams &P, cudaStream_t stream) {
  using Cfg = PtCfg<D_HEAD, PAIR>;
  auto k0 = kvd_prefill_attn_tc_kernel<D_HEAD, G, 0, PAIR>;
  auto k1 = kvd_prefill_attn_tc_kernel<D_HEAD, G, 1, PAIR>;
  static bool configured[64] = {};
  if (!configured[ctx->device & 63]) {
    cudaError_t e = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute(prefill attention)");
    configured[ctx->device & 63] = true;
  }
  const int tok = PT_ROWS / G;
  int tiles = (P.n_rows + tok - 1) / tok;
  if (PAIR) tiles = (tiles + 1) & ~1;  // whole pairs: a CTA whose tile lies past the last row has no rows to store
  return prefill_launch(ctx, ctx->dtype == 1 ? k1 : k0, tiles * P.n_kv, PT_THREADS, Cfg::SMEM_BYTES, PAIR ? 2 : 1, stream, P);
}

// Time a launch of CTAs of `tok` tokens would take: a CTA costs `per_cta` + `per_block` for every key block it walks, the
// CTAs start longest first, so an SM gets one of the first round, one of the reversed second round, and so on.  The
// positions are on the device; the host assumes the usual call, whose last row sits at the last key.
static float prefill_estimate(const kvd_ctx *ctx, const PrefillParams &P, int tok, float per_cta, float per_block) {
  const int tiles = (P.n_rows + tok - 1) / tok, total = tiles * P.n_kv, sms = ctx->num_sms;
  auto cost = [&](int i) {
    const int t0 = (tiles - 1 - i / P.n_kv) * tok, t1 = (t0 + tok < P.n_rows ? t0 + tok : P.n_rows) - 1;
    const int last = P.seg_hi - (P.n_rows - 1 - t1);
    int first = first_visible(P.seg_hi - (P.n_rows - 1 - t0), P.window);
    first = first < P.seg_lo ? P.seg_lo : first;
    return per_cta + per_block * static_cast<float>(last >= first ? last / PT_KEYS - first / PT_KEYS + 1 : 0);
  };
  float longest = 0.f;
  for (int m = 0; m < sms && m < total; ++m) {
    float sum = 0.f;
    for (int r = 0; r * sms < total; ++r) {
      const int i = r * sms + (r % 2 == 0 ? m : sms - 1 - m);
      if (i < total) sum += cost(i);
    }
    longest = sum > longest ? sum : longest;
  }
  return longest;
}

// Two tiles per CTA (d_head 128) or one.  Two serve more rows per clock but walk a block more slowly, so a call whose
// longest tiles set its time wants one, and one that keeps every SM busy for several rounds wants two.  Up to one round
// of single tiles: one.  Beyond four rounds: two.  Between: by estimate; the costs (us) were fitted to 102 launches of 1 to
// 27 rounds with groups of 1 to 8, windows of 0, 128 and 1024 and 0 to 7000 earlier keys (5 % rms), before the waits of
// both kernels became cheaper; the choices are right for what they cost now.  One / two tiles per CTA, us: 32 query on 8 KV
// heads, 600 tokens 13.4 / 19.6, 600 on 7000 169 / 134, 1300 33.8 / 31.2, 2500 89 / 75, 4096 198 / 151; 16 on 8, 1300 20.8 /
// 29.5, 1300 on 4000 106 / 97, 2500 49.0 / 49.6, 4096 101 / 75; 4 on 1, 8000 100 / 140, 8000 on 4000 180 / 205.  Two tiles
// whenever there is more than one round cost up to 1.5 times the time.  At d_head 64 the products are too short for two
// tiles: 294 tiles of a SmolLM2 layer 58 / 72 us.
static bool prefill_dual_pays(const kvd_ctx *ctx, const PrefillParams &P, int group) {
  const int tok = PT_ROWS / group;
  const long long tiles = static_cast<long long>((P.n_rows + tok - 1) / tok) * P.n_kv;
  if (tiles <= ctx->num_sms) return false;
  if (tiles > 4 * ctx->num_sms) return true;
  return prefill_estimate(ctx, P, 2 * tok, 10.4f, 1.07f) < prefill_estimate(ctx, P, tok, 6.0f, 0.74f);
}

// One tile on two CTAs: where every tile gets its own pair of SMs (beyond that the pairs would take turns) and the walk is
// long enough to pay for the second CTA's set-up.  Call alone, us, one tile per CTA or pair of tiles per pair / one tile on
// two CTAs, Gemma-3-4B layer: 16 tokens 7.5 / 10.9, 16 on 200 (4 blocks) 10.1 / 11.5, 290 13.2 / 12.1, 64 on 400 (8 blocks)
// 16.5 / 15.7, 64 on 1000 23.9 / 18.6, 600 18.5 / 14.6, 290 on 4000 66.6 / 41.2, 1100 on 4000 (72 tiles) 78.2 / 49.7;
// Qwen3-4B layer: 150 (3 blocks) 7.8 / 8.3, 64 on 400 11.7 / 10.4, 150 on 1000 18.7 / 15.0, 16 on 4000 49.5 / 31.4.
// (The positions are on the device; the host assumes the usual call, whose last row sits at the last key.)
static bool prefill_split_pays(const kvd_ctx *ctx, const PrefillParams &P, int group) {
  constexpr int LEAST_BLOCKS = 6;
  const int tok = PT_ROWS / group;
  const long long tiles = static_cast<long long>((P.n_rows + tok - 1) / tok) * P.n_kv;
  if (2 * tiles > ctx->num_sms) return false;
  int first = first_visible(P.seg_hi - (P.n_rows < tok ? P.n_rows : tok), P.window);
  first = first < P.seg_lo ? P.seg_lo : first;
  return P.seg_hi / PT_KEYS - first / PT_KEYS + 1 >= LEAST_BLOCKS;
}

template <int D_HEAD>
static kvd_status prefill_tc_group(kvd_ctx *ctx, const PrefillParams &P, int group, cudaStream_t stream) {
  // pairs where the K/V bytes per block bound the kernel (d_head = 256); at 128 the softmax does, and the hand-overs
  // across the pair cost more than the halved traffic returns (measured).  KVD_PREFILL_PAIR=0/1 asks for whole tiles on single
  // CTAs or pairs in calls of any length, for comparisons.
  static const char *env = getenv("KVD_PREFILL_PAIR");
  const bool pair = D_HEAD >= 128 && (env ? env[0] == '1' : D_HEAD == 256);
  if constexpr (D_HEAD >= 128) {
    if (!env && prefill_split_pays(ctx, P, group)) {
      switch (group) {
        case 1: return prefill_split_launch<D_HEAD, 1>(ctx, P, stream);
        case 2: return prefill_split_launch<D_HEAD, 2>(ctx, P, stream);
        case 3: return prefill_split_launch<D_HEAD, 3>(ctx, P, stream);
        case 4: return prefill_split_launch<D_HEAD, 4>(ctx, P, stream);
        case 8: return prefill_split_launch<D_HEAD, 8>(ctx, P, stream);
        default: return KVD_ERR_SHAPE;
      }
    }
    if (pair) {
      switch (group) {
        case 1: return prefill_tc_launch<D_HEAD, 1, true>(ctx, P, stream);
        case 2: return prefill_tc_launch<D_HEAD, 2, true>(ctx, P, stream);
        case 3: return prefill_tc_launch<D_HEAD, 3, true>(ctx, P, stream);
        case 4: return prefill_tc_launch<D_HEAD, 4, true>(ctx, P, stream);
        case 8: return prefill_tc_launch<D_HEAD, 8, true>(ctx, P, stream);
        default: return KVD_ERR_SHAPE;
      }
    }
  }
  if constexpr (D_HEAD == 128) {
    if (prefill_dual_pays(ctx, P, group)) {
      switch (group) {
        case 1: return prefill_dual_launch<D_HEAD, 1>(ctx, P, stream);
        case 2: return prefill_dual_launch<D_HEAD, 2>(ctx, P, stream);
        case 3: return prefill_dual_launch<D_HEAD, 3>(ctx, P, stream);
        case 4: return prefill_dual_launch<D_HEAD, 4>(ctx, P, stream);
        case 8: return prefill_dual_launch<D_HEAD, 8>(ctx, P, stream);
        default: return KVD_ERR_SHAPE;
      }
    }
  }
  switch (group) {
    case 1: return prefill_tc_launch<D_HEAD, 1, false>(ctx, P, stream);
    case 2: return prefill_tc_launch<D_HEAD, 2, false>(ctx, P, stream);
    case 3: return prefill_tc_launch<D_HEAD, 3, false>(ctx, P, stream);
    case 4: return prefill_tc_launch<D_HEAD, 4, false>(ctx, P, stream);
    case 8: return prefill_tc_launch<D_HEAD, 8, false>(ctx, P, stream);
    default: return KVD_ERR_SHAPE;
  }
}

kvd_status launch_prefill_tc(kvd_ctx *ctx, const PrefillParams &P, int d_head, int group, cudaStream_t stream) {
  switch (d_head) {
    case 64: return prefill_tc_group<64>(ctx, P, group, stream);
    case 128: return prefill_tc_group<128>(ctx, P, group, stream);
    case 256: return prefill_tc_group<256>(ctx, P, group, stream);
    default: return KVD_ERR_SHAPE;
  }
}

}  // namespace kvd
