// Projection of a few rows (at most 64): the K/V of a decode step's new tokens when nothing is recomputed in
// the same call, and the dense products of a decoder block at decode batch sizes.
//
//   Y[M <= 64, N] = X[M, K] * W'      W' K-major, the products and the finishing of kvd_recompute.cu
//
// Bound: reading W' once (N * K * 2 bytes).  The 256-row tile of the recompute kernel spends a full tile's MMA
// time (512 clocks per 64 channels) on rows that are not there and cuts N into 256-column tiles, i.e. 8 to 10
// CTA pairs for the models' projections.  Here a tile is as narrow as it takes to give every SM one (a multiple
// of 8 columns, RW_MIN_TILE at least), so that all SMs pull weights at once.
//
// The MMA has 64 rows however few of them are rows of X; only those are loaded, the descriptor's other rows are whatever
// lies behind them in shared memory, and their accumulators (lanes of tensor memory) are never read.
//
// The bits are those of the recompute kernel: an output element is one accumulator that takes the same K = 16
// steps in the same ascending order, and the finishing below repeats that kernel's operations and their order
// (row statistic, key norm, rotation, rounding).
//
// Measured (B200, one bf16 row, time of the launch alone): 2560 -> 262144 columns 323 us with the 256-row tiles, 197 us
// here (6.8 TB/s of weights); 2560 -> 20480 43 and 23.5 us; 10240 -> 2560 54 and 20.7 us; 2560 -> 2048 20 and 10.7 us; K and
// V of a Gemma-3-4B layer 25.6 and 12.9 us.  Short products are bound by launch, first-load latency and, where K is
// long, by the chain of K / 16 dependent MMAs (24 clocks each alone; 36 in this kernel before the issuer asked for a stage
// ahead of its end, 27 since: in a chain of launches 10240 -> 2560 15.3 -> 13.3 us, with 24 rows 22.7 -> 20.0).  The operands the other way round (weights as the M
// of the MMA, 64 columns per CTA) measured 282, 38 and 44 us: too few CTAs for the narrow products.
//
// Weights never change after they were prepared, so the loads of the first stages are issued before the
// dependency wait: with programmatic launches they run under the tail of the preceding kernel.
//
// Warps: 0 producer (one lane), 1 MMA issuer (one lane) and tensor-memory owner, 2-9 row statistics, of these
// 4-7 the epilogue.  Plain products walk over tiles (two accumulators); key/value projections
// have one 32-column tile per CTA, the d_head / 32 CTAs of a head form a cluster and exchange their accumulators where
// the key norm runs over the whole head in one fixed order or the half-split rotation pairs columns of different tiles.
// What the end of a CTA waits for is latency: the columns travel by st.async, 16 bytes a lane, and count on the receiver's
// barrier; two lanes take a row's norm; positions, rotation and scale of the keys are fetched while the products run.  (One
// thread per row storing to every CTA, a cluster barrier, then the norm, then the tables: 2.6 us behind the last product;
// one row of a Gemma-3-4B layer in a chain 6.5 -> 5.6 us, three 6.2 -> 5.5.)
#include <string.h>

#include <type_traits>

#include "kvd_internal.h"
#include "kvd_ptx.cuh"

namespace kvd {

constexpr int RW_THREADS = 320;

// Four K = 16 steps of one k block: D[64 rows][columns of the tile] += X[64 x 64] W'^T[64 x columns].
__device__ __forceinline__ void umma_kblock(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                            uint32_t acc_first) {
  asm volatile(
      "{\n\t"
      ".reg .pred p, t;\n\t"
      ".reg .b64 da, db;\n\t"
      ".reg .b32 la, lb;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "setp.eq.b32 t, 0, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t"
      "add.u32 la, %1, 2;\n\t"
      "add.u32 lb, %2, 2;\n\t"
      "mov.b64 da, {la, %3};\n\t"
      "mov.b64 db, {lb, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, t;\n\t"
      "add.u32 la, %1, 4;\n\t"
      "add.u32 lb, %2, 4;\n\t"
      "mov.b64 da, {la, %3};\n\t"
      "mov.b64 db, {lb, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, t;\n\t"
      "add.u32 la, %1, 6;\n\t"
      "add.u32 lb, %2, 6;\n\t"
      "mov.b64 da, {la, %3};\n\t"
      "mov.b64 db, {lb, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, t;\n\t"
      "}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc_first)
      : "memory");
}

// D_HEAD = 0: a plain product, every column scaled by the row factor and stored.  D_HEAD > 0: key and value heads.
template <int D_HEAD, int DT>
__global__ void __launch_bounds__(RW_THREADS, 2)
kvd_rows_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                const __grid_constant__ RowsParams p) {
  constexpr bool HEADS = D_HEAD > 0;
  constexpr int CL = HEADS ? D_HEAD / RW_HEAD_TILE : 1;  // CTAs of a head
  constexpr int LD = HEADS ? D_HEAD + 4 : 0;             // floats between the rows of s_y
  extern __shared__ __align__(1024) uint8_t rw_smem[];
  if ((smem_u32(rw_smem) & 1023u) != 0u) {  // the 128-byte swizzle is anchored at 1024-byte boundaries
    if (threadIdx.x == 0) atomicOr(p.status, STATUS_TIMEOUT);
    return;
  }
  const int stages = p.stages, kbs = p.stage_kb, tile = p.tile;
  const uint32_t x_kb = static_cast<uint32_t>(p.nr) * 128u, w_kb = static_cast<uint32_t>(tile) * 128u;  // bytes per k block
  const uint32_t stage_bytes = kbs * (x_kb + w_kb), w_off = kbs * x_kb;
  uint8_t *tail = rw_smem + p.tail_off;  // behind the ring and the rows its last descriptor spans
  uint64_t *bars = reinterpret_cast<uint64_t *>(tail);
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + RW_BARS);
  volatile int *s_abort = reinterpret_cast<volatile int *>(s_tmem + 1);
  float *s_rstd = reinterpret_cast<float *>(s_tmem + 8);
  float *s_kscale = s_rstd + RW_MAX_ROWS;
  float *s_y = s_kscale + RW_MAX_ROWS;  // heads: accumulators of the whole head, [row][LD]
  const uint32_t ring = smem_u32(rw_smem), bar_base = smem_u32(bars);
  auto bar_full = [&](int s) { return bar_base + 8u * s; };
  auto bar_empty = [&](int s) { return bar_base + 8u * (RW_MAX_STAGES + s); };
  auto bar_tmem_full = [&](int a) { return bar_base + 8u * (2 * RW_MAX_STAGES + a); };
  auto bar_tmem_empty = [&](int a) { return bar_base + 8u * (2 * RW_MAX_STAGES + 2 + a); };
  const uint32_t bar_head = bar_base + 8u * (2 * RW_MAX_STAGES + 4);  // keys: the other CTAs' columns of the head
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const unsigned long long tmo = p.timeout_ns;
  const int steps = (p.num_k_blocks + kbs - 1) / kbs;  // stages of a tile
  const int block = static_cast<int>(blockIdx.x), blocks = static_cast<int>(gridDim.x);
  const int my_tiles = (p.n_tiles - block + blocks - 1) / blocks;
  const int head_col = block * RW_HEAD_TILE;     // heads: the CTA's first column
  const bool key = HEADS && head_col < p.k_cols;
  const bool exchange = key && (p.qk_norm || p.rope_half);  // what it makes of its columns depends on other CTAs' columns
  // heads: the last part's row of this thread (half a warp per row) and what the rotation of its two columns takes, fetched
  // by warps 2 to 9 while the products run
  const int last_row = 2 * ((warp + 8) % 10) + (lane >> 4), head_c = head_col % (HEADS ? D_HEAD : 1) + 2 * (lane & 15);
  struct Turn {
    float cs[2], sn[2], ga[2], gb[2];
  } turn = {};
  auto position = [&](int r) {
    const int pos = p.positions[r];
    if (pos >= 0 && pos < p.max_pos) return pos;
    atomicOr(p.status, STATUS_POSITION);
    return pos < 0 ? 0 : p.max_pos - 1;
  };
  auto fetch_turn = [&](int pos) {
    if constexpr (HEADS) {
      constexpr int HALF = D_HEAD / 2;
      const float2 *t_hi = p.rope_hi + static_cast<size_t>(pos >> ROPE_LO_BITS) * HALF;
      const float2 *t_lo = p.rope_lo + (pos & (ROPE_LO_SIZE - 1));
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = p.rope_half ? (head_c + j) % HALF : head_c / 2;  // pair (i, i + HALF), or the columns' own
        const float2 h = __ldg(t_hi + i), l = __ldg(t_lo + i * ROPE_LO_SIZE);
        turn.cs[j] = fmaf(h.x, l.x, -h.y * l.y);
        turn.sn[j] = fmaf(h.y, l.x, h.x * l.y);
        turn.ga[j] = p.gamma_k ? __ldg(p.gamma_k + (p.rope_half ? i : head_c)) : 1.0f;
        turn.gb[j] = p.gamma_k ? __ldg(p.gamma_k + (p.rope_half ? i + HALF : head_c + 1)) : 1.0f;
      }
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_tmem_full(a), 1);
      mbar_init(bar_tmem_empty(a), 4);  // one arrival per epilogue warp
    }
    *s_abort = 0;
    if (HEADS) mbar_init(bar_head, 1);
    fence_mbar_init();
    if (exchange) mbar_arrive_expect_tx(bar_head, (CL - 1) * p.n_rows * RW_HEAD_TILE * 4);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem), p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  if (CL > 1) cluster_sync_all();  // (also: every CTA of the head runs before anyone writes into its shared memory)
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  // Only now, with the tensor memory in hand: the allocation is a wait without a limit, and a dependent let in before it
  // could take the columns this CTA waits for, and then wait for this kernel's end.
  grid_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    const int total = my_tiles * steps, pre = total < stages ? total : stages;
    if (elect_one()) {
      for (int i = 0; i < pre; ++i) {
        mbar_arrive_expect_tx(bar_full(i), stage_bytes);
        tma_load_3d(ring + i * stage_bytes + w_off, &tmap_w, bar_full(i), 0, (block + i / steps * blocks) * tile, i % steps * kbs);
      }
    }
    grid_dependency_wait();  // the rows may come from the preceding kernel
    if (elect_one()) {
      for (int i = 0; i < pre; ++i) tma_load_3d(ring + i * stage_bytes, &tmap_x, bar_full(i), 0, 0, i % steps * kbs);
      int issued = pre, s = 0, k = pre % steps, col = (block + pre / steps * blocks) * tile;
      uint32_t ph = 0;  // parity of the phase of `empty` that frees stage s for its next fill
      for (; issued < total; ++issued) {
        if (!mbar_wait(bar_empty(s), ph, s_abort, tmo)) {
          raise(p.status, STATUS_TIMEOUT, s_abort);
          break;
        }
        mbar_arrive_expect_tx(bar_full(s), stage_bytes);
        tma_load_3d(ring + s * stage_bytes + w_off, &tmap_w, bar_full(s), 0, col, k * kbs);
        tma_load_3d(ring + s * stage_bytes, &tmap_x, bar_full(s), 0, 0, k * kbs);
        if (++k == steps) {
          k = 0;
          col += blocks * tile;
        }
        if (++s == stages) {
          s = 0;
          ph ^= 1u;
        }
      }
      // Leave no copy in flight: wait (bounded) for the last fill of every stage.  Always, and longer than the MMA issuer
      // waits: that thread may give up after this one has issued everything, and then nobody else watches the copies.
      // (In a launch that runs its course the issuer waits for the same fills.)
      const unsigned long long t0 = globaltimer_ns();
      for (int b = 0; b < stages && b < issued; ++b) {
        const uint32_t par = static_cast<uint32_t>((issued - 1 - b) / stages) & 1u;
        while (!mbar_try_wait(bar_full(b), par))
          if (globaltimer_ns() - t0 > tmo + 100000000ull) break;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    grid_dependency_wait();  // (the bounded waits below start when the rows can be loaded)
    if (elect_one()) {  // (24 clocks per MMA; 48 in a branch on the lane number)
      const uint32_t idesc = DT == 1 ? umma_idesc_f16_f32(RW_MMA_ROWS, tile) : umma_idesc_bf16_f32(RW_MMA_ROWS, tile);
      constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);  // as in kvd_recompute.cu
      int s = 0;
      uint32_t ph = 0, ready = 0;  // ready: stage s is known to have landed
      bool ok = true;
      for (int t = 0; ok && t < my_tiles; ++t) {
        const int a = t & 1;
        if (!mbar_wait(bar_tmem_empty(a), ((t >> 1) & 1u) ^ 1u, s_abort, tmo)) {
          raise(p.status, STATUS_TIMEOUT, s_abort);
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem_base + a * (p.tmem_cols / 2);
        int left = p.num_k_blocks;
        for (int k = 0; k < steps; ++k) {
          if (!ready && !mbar_wait(bar_full(s), ph, s_abort, tmo)) {
            raise(p.status, STATUS_TIMEOUT, s_abort);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t xa = ((ring + s * stage_bytes) >> 4) | (1u << 16), wb = ((ring + s * stage_bytes + w_off) >> 4) | (1u << 16);
          const uint32_t x_step = x_kb >> 4, w_step = w_kb >> 4, empty = bar_empty(s);
          if (++s == stages) {
            s = 0;
            ph ^= 1u;
          }
          const int n = left < kbs ? left : kbs;
          umma_kblock(d, xa, wb, desc_hi, idesc, k != 0 ? 1u : 0u);
          // The tensor cores hold few MMAs ahead of the one they work on, and a barrier answers late beside their reads of
          // shared memory: asked for between two stages, the next one's state cost 250 clocks of idle tensor cores.
          ready = mbar_test_wait(bar_full(s), ph);
          if (n == 8) {
#pragma unroll
            for (int b = 1; b < 8; ++b) umma_kblock(d, xa + b * x_step, wb + b * w_step, desc_hi, idesc, 1u);
          } else {
            for (int b = 1; b < n; ++b) umma_kblock(d, xa + b * x_step, wb + b * w_step, desc_hi, idesc, 1u);
          }
          left -= n;
          umma_commit(empty);
        }
        if (ok) umma_commit(bar_tmem_full(a));
      }
    }
  } else {
    // ------------------------------------------------------------------ row statistics (Eq. 2)
    grid_dependency_wait();
    const int w8 = warp - 2;
    if (p.sumsq != nullptr) {
      const int row = threadIdx.x - 64;
      if (row < p.n_rows) s_rstd[row] = 1.0f / sqrtf(p.sumsq[row] * p.inv_k + p.rms_eps);
    } else {
      // STORE_RESIDUAL in the same launch (kvd_decode_step_kv): the first CTA writes the rows it reads into the
      // store slots the host assigned to them
      const bool append = HEADS && p.append_rows != nullptr && block == 0;
      // R rows of a warp side by side, B loads of each in flight: one round trip for the usual width and up to 8 rows
      auto take = [&](auto r_c, auto b_c) {
        constexpr int R = decltype(r_c)::value, B = decltype(b_c)::value;
#pragma unroll 1
        for (int g = w8; R * g < p.n_rows; g += 8) {
          const uint4 *src[R];
          uint4 *dst[R];
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int r = R * g + i;
            src[i] = p.rows + static_cast<size_t>(r < p.n_rows ? r : p.n_rows - 1) * p.row_chunks;
            dst[i] = nullptr;
            // (checking build: the slot lies inside the store)
            if (append && r < p.n_rows && KVD_BOUNDS_OK(p.append_slot[r] >= 0 && p.append_slot[r] < p.store_slots, p.status))
              dst[i] = p.append_rows + static_cast<size_t>(p.append_slot[r]) * p.row_chunks;
          }
          float ss[R];
          warp_rows_sumsq<R, B, HEADS, DT>(src, dst, p.row_chunks, lane, ss);
          float mine = ss[0];
#pragma unroll
          for (int i = 1; i < R; ++i) mine = lane == i ? ss[i] : mine;
          const int r = R * g + lane;
          if (lane < R && r < p.n_rows) {
            s_rstd[r] = 1.0f / sqrtf(mine * p.inv_k + p.rms_eps);
            if (append && KVD_BOUNDS_OK(p.append_slot[r] >= 0 && p.append_slot[r] < p.store_slots, p.status)) {
              p.append_sumsq[p.append_slot[r]] = mine;
              p.append_pos[p.append_slot[r]] = p.positions[r];
            }
          }
        }
      };
      if (p.n_rows <= 8) take(std::integral_constant<int, 1>(), std::integral_constant<int, 10>());
      else take(std::integral_constant<int, 2>(), std::integral_constant<int, 5>());
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (key && last_row < p.n_rows) fetch_turn(position(last_row));
    if (warp >= 4 && warp < 8) {
      // ---------------------------------------------------------------- epilogue
      // (M = 64: rows 16 q .. 16 q + 15 are lanes 0-15 of tensor memory quarter q)
      const int quarter = warp & 3, row = quarter * 16 + lane;
      const bool valid = lane < 16 && row < p.n_rows, busy = quarter * 16 < p.n_rows;  // busy: warp-uniform
      const uint32_t rank = CL > 1 ? cluster_ctarank() : 0u;
      const float rstd = valid ? s_rstd[row] : 0.f;
      for (int t = 0; t < my_tiles; ++t) {
        const int a = t & 1, col0 = (block + t * blocks) * tile;
        if (!warp_wait(bar_tmem_full(a), (t >> 1) & 1u, s_abort, tmo, lane)) {
          raise(p.status, STATUS_TIMEOUT, s_abort);
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + a * (p.tmem_cols / 2);
        // (checking build: the tile's columns exist; otherwise none is stored)
        const int cols = !KVD_BOUNDS_OK(col0 >= 0 && col0 < p.n_cols && col0 % tile == 0, p.status) ? 0 : p.n_cols - col0 < tile ? p.n_cols - col0 : tile;
        if constexpr (HEADS) {
          if (busy) {
            uint32_t v[RW_HEAD_TILE];
            tmem_ld_x32(acc, v);
            tmem_wait_ld();
            float *mine = s_y + static_cast<int>(rank) * RW_HEAD_TILE;
            if (valid) {
#pragma unroll
              for (int j = 0; j < RW_HEAD_TILE; j += 4) *reinterpret_cast<uint4 *>(mine + row * LD + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
            if (exchange) {  // keys: the whole head goes to each of its CTAs, (CL - 1) x 8 pieces of 16 bytes a row
              __syncwarp();
              for (int i = lane; i < static_cast<int>(CL - 1) * 8; i += 32) {
                const uint32_t to = (rank + 1 + i / 8) % CL, bar = map_to_cta(bar_head, to);
                for (int r = quarter * 16; r < p.n_rows && r < quarter * 16 + 16; ++r) {
                  const float *src = mine + r * LD + i % 8 * 4;
                  const uint4 y = *reinterpret_cast<const uint4 *>(src);
                  st_async_v4(map_to_cta(smem_u32(src), to), bar, y.x, y.y, y.z, y.w);
                }
              }
            }
          }
        } else {
          __nv_bfloat16 *dst = p.v_out + static_cast<size_t>(row) * p.out_stride + col0;
          int c = 0;
          for (; busy && c + 32 <= cols; c += 32) {
            uint32_t v[32], o[16];
            tmem_ld_x32(acc + c, v);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = pack_out<DT>(__uint_as_float(v[2 * j]) * rstd, __uint_as_float(v[2 * j + 1]) * rstd);
            if (valid) store_row_piece<4>(dst + c, o, p.wide_store != 0);
          }
          for (; busy && c < cols; c += 8) {
            uint32_t v[8], o[4];
            tmem_ld_x8(acc + c, v);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = pack_out<DT>(__uint_as_float(v[2 * j]) * rstd, __uint_as_float(v[2 * j + 1]) * rstd);
            if (valid) store_row_piece<1>(dst + c, o, false);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tmem_empty(a));
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, p.tmem_cols);
  }
  if constexpr (HEADS) {
    // ------------------------------------------------------------------ key norm, rotation, stores: all warps
    // (No CTA leaves before every CTA of the head has sent its columns, and each waits for those it is sent, also behind
    // an abort: nothing arrives in the shared memory of a CTA that is gone.)
    cluster_arrive_relaxed();
    auto columns_within = [&](unsigned long long limit_ns) -> bool {
      int ok = 1;
      if (lane == 0) {
        const unsigned long long t0 = globaltimer_ns();
        while (!mbar_try_wait_cluster(bar_head, 0))
          if (globaltimer_ns() - t0 > limit_ns) {
            ok = 0;
            break;
          }
      }
      return __shfl_sync(0xffffffffu, ok, 0) != 0;
    };
    const bool got = !exchange || columns_within(tmo);
    if (!got) raise(p.status, STATUS_TIMEOUT, s_abort);
    __syncwarp();
    constexpr int HALF = D_HEAD / 2;
    // two lanes per row: four chains (columns j mod 4) in ascending order, two-wide: the order of the recompute kernel
    if (warp * 16 < p.n_rows) {
      const int r = threadIdx.x / 2 < p.n_rows ? threadIdx.x / 2 : p.n_rows - 1, half = threadIdx.x & 1;
      const float rstd = s_rstd[r];
      float kscale = rstd;
      if (key && p.qk_norm) {
        uint64_t ss2 = 0ull;
        const uint64_t rstd2 = pack2(rstd, rstd);
#pragma unroll 16
        for (int c = 2 * half; c < D_HEAD; c += 4) {
          const float2 y = *reinterpret_cast<const float2 *>(s_y + r * LD + c);
          const uint64_t v = fmul2(pack2(y.x, y.y), rstd2);
          ss2 = ffma2(v, v, ss2);
        }
        float s0, s1;
        unpack2(ss2, s0, s1);
        const float mine = s0 + s1, ss = mine + __shfl_xor_sync(0xffffffffu, mine, 1);
        kscale = rstd * (1.0f / sqrtf(ss * (1.0f / D_HEAD) + p.qk_eps));
      }
      s_kscale[r] = kscale;
    }
    __syncthreads();
    const bool whole = *s_abort == 0;
    for (int r = last_row; whole && r < p.n_rows; r += 2 * (RW_THREADS / 32)) {
      // (checking build: this CTA's columns lie inside the key or the value heads)
      if (!KVD_BOUNDS_OK(head_col + RW_HEAD_TILE <= (key ? p.k_cols : p.n_cols) && r < RW_MAX_ROWS, p.status)) continue;
      const float *y = s_y + r * LD;
      const float ks = s_kscale[r];
      const int c = head_c;
      uint32_t o;
      if (!key) {
        o = pack_out<DT>(y[c] * ks, y[c + 1] * ks);
      } else {
        if (warp < 2 || r != last_row) fetch_turn(position(r));
        if (!p.rope_half) {
          const float a = y[c] * ks * turn.ga[0], b = y[c + 1] * ks * turn.gb[0];
          o = pack_out<DT>(fmaf(a, turn.cs[0], -b * turn.sn[0]), fmaf(a, turn.sn[0], b * turn.cs[0]));
        } else {
          float v[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int i = (c + j) % HALF;  // pair (i, i + HALF)
            const float a = y[i] * ks * turn.ga[j], b = y[i + HALF] * ks * turn.gb[j];
            v[j] = c < HALF ? fmaf(a, turn.cs[j], -b * turn.sn[j]) : fmaf(a, turn.sn[j], b * turn.cs[j]);
          }
          o = pack_out<DT>(v[0], v[1]);
        }
      }
      __nv_bfloat16 *dst = (key ? p.k_out + (head_col / D_HEAD) * D_HEAD : p.v_out + (head_col - p.k_cols) / D_HEAD * D_HEAD) +
                           static_cast<size_t>(r) * p.out_stride + c;
      *reinterpret_cast<uint32_t *>(dst) = o;
    }
    __syncwarp();
    cluster_wait();
    // Every CTA has sent by now what it sends, but its arrival does not say that it has landed: a CTA that has not seen all
    // columns stays for as long as that could take.
    if (!got) columns_within(200000ull);
  }
}

template <int D_HEAD, int DT>
static kvd_status launch_rows_impl(kvd_ctx *ctx, const CUtensorMap &tmap_w, const CUtensorMap &tmap_x, RowsParams &p, cudaStream_t stream) {
  auto kern = kvd_rows_kernel<D_HEAD, DT>;
  constexpr int CL = D_HEAD > 0 ? D_HEAD / RW_HEAD_TILE : 1;
  static bool configured[64] = {};
  if (!configured[ctx->device & 63]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RW_SMEM_MAX);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute(rows)");
    configured[ctx->device & 63] = true;
  }
  const RowsRing ring = rows_ring(p.nr, p.tile, p.stage_kb, D_HEAD, (p.num_k_blocks + p.stage_kb - 1) / p.stage_kb * ((p.n_tiles + ctx->num_sms - 1) / ctx->num_sms));
  p.stages = ring.stages;
  p.tail_off = ring.tail_off;
  p.tmem_cols = 64;  // two accumulators; the epilogue reads 32 columns at once
  while (p.tmem_cols < 2 * p.tile) p.tmem_cols *= 2;
  const int grid = D_HEAD > 0 || p.n_tiles < ctx->num_sms ? p.n_tiles : ctx->num_sms;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(RW_THREADS, 1, 1);
  cfg.dynamicSmemBytes = ring.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = (serial_launch_mask() & 1) ? 0 : 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL > 1 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmap_w, tmap_x, p);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "launch rows");
  ctx->launches += 1;
  if (D_HEAD > 0) ctx->few_rows.set(ctx->launches, stream);
  return KVD_OK;
}

// 3-D map [k block][row][64 channels] of a K-major 16-bit matrix: a box is stage_kb k blocks of box_rows rows.
static kvd_status encode_kblocks(kvd_ctx *ctx, CUtensorMap *map, const void *base, int k, int rows, int box_rows, int stage_kb) {
  cuuint64_t dims[3] = {RC_BLOCK_K, static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(k / RC_BLOCK_K)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(k) * 2, RC_BLOCK_K * 2};
  cuuint32_t box[3] = {RC_BLOCK_K, static_cast<cuuint32_t>(box_rows), static_cast<cuuint32_t>(stage_kb)};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = ctx->encode(map, ctx->dtype == KVD_DTYPE_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                           const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    ctx->last_error = "cuTensorMapEncodeTiled (k blocks) failed: " + std::to_string(static_cast<int>(r));
    return KVD_ERR_CUDA;
  }
  return KVD_OK;
}

// Columns per tile of a plain product: one tile per SM, or as few equal rounds of tiles of at most 256 columns.
static int rows_tile(const kvd_ctx *ctx, int n_cols) {
  const int rounds = (n_cols + 256 * ctx->num_sms - 1) / (256 * ctx->num_sms);
  const int t = ((n_cols + rounds * ctx->num_sms - 1) / (rounds * ctx->num_sms) + 7) / 8 * 8;
  return t < RW_MIN_TILE ? RW_MIN_TILE : t;
}
kvd_status prepare_rows_map(kvd_ctx *ctx, LayerState &ls, int k, int n_cols, bool heads) {
  ls.rows_tile = heads ? RW_HEAD_TILE : rows_tile(ctx, n_cols);
  kvd_status st = KVD_OK;
  for (int many = 0; st == KVD_OK && many < 2; ++many)
    st = encode_kblocks(ctx, &ls.tmap_rows[many], ls.wt, k, n_cols, ls.rows_tile, rows_stage_kb(ls.rows_tile, many != 0));
  return st;
}

kvd_status launch_rows(kvd_ctx *ctx, const LayerState &ls, int k, RowsParams &p, bool heads, cudaStream_t stream) {
  p.nr = (p.n_rows + 7) / 8 * 8;
  p.num_k_blocks = k / RC_BLOCK_K;
  p.tile = ls.rows_tile;
  const bool many = p.nr > RW_FEW_ROWS;
  p.stage_kb = rows_stage_kb(p.tile, many);
  if (p.tile % 16 != 0) p.wide_store = 0;  // a tile has to start at a 32-byte boundary for 32-byte stores
  p.n_tiles = (p.n_cols + p.tile - 1) / p.tile;
  CUtensorMap tmap_x;
  kvd_status st = encode_kblocks(ctx, &tmap_x, p.rows, k, p.n_rows, p.nr, p.stage_kb);
  if (st != KVD_OK) return st;
  const CUtensorMap &w = ls.tmap_rows[many ? 1 : 0];
  if (!heads) return launch_rows_impl<0, 0>(ctx, w, tmap_x, p, stream);
  const bool half = ctx->dtype == KVD_DTYPE_F16;
  switch (ctx->desc.d_head) {
    case 64: return half ? launch_rows_impl<64, 1>(ctx, w, tmap_x, p, stream) : launch_rows_impl<64, 0>(ctx, w, tmap_x, p, stream);
    case 128: return half ? launch_rows_impl<128, 1>(ctx, w, tmap_x, p, stream) : launch_rows_impl<128, 0>(ctx, w, tmap_x, p, stream);
    case 256: return half ? launch_rows_impl<256, 1>(ctx, w, tmap_x, p, stream) : launch_rows_impl<256, 0>(ctx, w, tmap_x, p, stream);
    default: return KVD_ERR_SHAPE;
  }
}

}  // namespace kvd
