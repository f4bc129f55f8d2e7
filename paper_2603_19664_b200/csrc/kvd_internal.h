// Host-side context and the parameter blocks passed to the kernels.  Internal to the library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

#include "../../include/kvd.h"
#include "kvd_launch_mark.h"
#include "kvd_positions.h"
#include "kvd_rows_ring.h"

namespace kvd {

// device status word bits (written by kernels with atomicOr, read by kvd_poll_status)
constexpr int STATUS_TIMEOUT = 1;
constexpr int STATUS_POSITION = 2;
constexpr int STATUS_BOUNDS = 4;  // checking build: an index test failed (the access was skipped)

// Index tests of the checking build (-DKVD_CHECK): `if (KVD_BOUNDS_OK(cond, status)) access;`.  A failed test
// records STATUS_BOUNDS and yields false, so the access is skipped; the release build compiles the test away.
#ifdef KVD_CHECK
#define KVD_BOUNDS_OK(cond, status) ((cond) ? true : ((status) != nullptr ? (atomicOr((status), kvd::STATUS_BOUNDS), false) : false))
#else
#define KVD_BOUNDS_OK(cond, status) (true)
#endif

constexpr int ROPE_LO_BITS = 4;  // position = hi * 16 + lo; one table per part
constexpr int ROPE_LO_SIZE = 1 << ROPE_LO_BITS;

// ------------------------------------------------------------------------------ recompute GEMM
constexpr int RC_BLOCK_M = 128;
constexpr int RC_BLOCK_K = 64;
// caller rows up to this count have their statistics taken inside the recompute kernel (its four
// statistics warps cover them under the main loop of one tile pair); more rows get a kernel of their own
constexpr int RC_INLINE_STAT_ROWS = 64;
constexpr int RC_TRACE_TILES = 8;    // tiles per CTA recorded when a trace buffer is attached
constexpr int RC_TRACE_FIELDS = 16;  // int64 slots per (CTA, tile); see kvd_set_trace
constexpr int RC_THREADS = 320;  // warp 2 TMA, warp 3 MMA, warps 0,1,8,9 row statistics, warps 4-7 epilogue
constexpr int RC_THREADS_8 = 384;  // with two epilogue groups: warps 0,1 row statistics, 4-7 and 8-11 epilogue (168 registers, as with 320)

// store slots of the rows of kvd_checkpoint_residual_step (one new row per sequence of a batch)
struct CkptSlots {
  long long slot[KVD_MAX_STORE_RANGES];
};

constexpr int RC_MAX_JOBS = 65;  // row sources per launch: up to 64 store ranges and one caller buffer

// One source of rows inside a launch.  Jobs own consecutive runs of 256-row blocks.
struct RcJob {
  int mb_start;  // first 256-row block of this job in the launch
  int n;         // rows
  int row0;      // first row: index into the store slab, or 0 for a caller buffer
  int slab;      // store slab (sequence slot of this layer), or -1: rows come from the caller's buffer
  const int32_t *positions;  // [n]
  const float *sumsq;        // [n] sum of squares of each row (store ranges), nullptr for the caller's rows
  const float *scale;        // [n] FP8 store: the rows' quantisation scales; nullptr for bf16 rows
  __nv_bfloat16 *k_out;      // row m of the job at k_out + m * out_row_stride
  __nv_bfloat16 *v_out;
};

struct RecomputeParams {
  int n_jobs;
  int num_k_blocks;  // d_hidden / 64
  int num_m_blocks;  // over all jobs
  int num_n_blocks;
  int unit_tiles, whole_tiles, parts, clusters;  // set by schedule_recompute
  int k_cols;  // n_kv * d_head: fused columns below this index are keys, the rest values
  long long out_row_stride;
  float inv_d_hidden;
  float rms_eps;
  int qk_norm;
  float qk_eps;
  int rope_style;
  const float2 *rope_hi;  // [n_hi][d_head/2] (cos, sin) of (pos & ~15) * freq_i
  const float2 *rope_lo;  // [d_head/2][16]   (cos, sin) of (pos & 15) * freq_i, pair-major
  int max_pos;            // positions must be in [0, max_pos)
  const float *gamma_k;   // [d_head] fp32 or nullptr
  int *status;
  unsigned long long timeout_ns;
  long long *trace;  // nullptr unless a trace buffer is attached
  const __nv_bfloat16 *ext_rows;  // the caller's rows (job with slab < 0), [n][d_hidden]
  int row_chunks;                 // d_hidden / 8: 16-byte chunks per row
  int wide_store;                 // outputs are 32-byte aligned: 32-byte stores
  const float *w_scale;           // FP8 variant: the weight matrix's quantisation scale (one float), else nullptr
  int store_rows;                 // rows per (layer, sequence) slab of the store (checking build)
  long long rows_out_stride;      // row stride of the caller rows' K/V outputs (the store ranges use out_row_stride)
  // STORE_RESIDUAL riding in the launch (kvd_decode_step_kv): caller row i is also written to slot append_slot[i]
  // of the store (rows, position, statistic), by the statistics warps that read it anyway
  int append_n;                   // 0: nothing is appended
  uint4 *append_rows;             // the store's rows, 16-byte chunks; slot s at append_rows + s * row_chunks
  int32_t *append_pos;
  float *append_sumsq;
  long long append_slot[RC_INLINE_STAT_ROWS];
  RcJob jobs[RC_MAX_JOBS];
};

// Fused recompute + attention (the recomputed K/V of a store range are consumed inside the kernel and
// never written): per job, the query of the range's sequence and where its partials go.
struct RcAttend {
  const __nv_bfloat16 *q;  // [n_q][d_head] of the job's sequence; nullptr: plain job, K and V are stored
  int q_pos;               // position of the query
  int lo_pos;              // first visible position (sliding window), 0 without a window
  int part_base;           // slot of the job's first 256-row block in the partial arrays
  int reserved;
};
struct FusedParams {
  float *part_o;   // [slot][n_q][d_head] unnormalised outputs
  float *part_ml;  // [slot][n_q][2] (max in log2 units, sum)
  int n_q;
  float scale_log2e;
  RcAttend att[RC_MAX_JOBS];
};
struct NoFusedParams {};

// ------------------------------------------------------------------------------ projection of a few rows
static_assert(RW_MAX_ROWS == RC_INLINE_STAT_ROWS, "rows of a call whose statistics are taken in the kernel");
struct RowsParams {
  const uint4 *rows;           // [n_rows][row_chunks]
  const int32_t *positions;    // [n_rows] (heads)
  const float *sumsq;          // [n_rows], or nullptr: taken from the rows
  __nv_bfloat16 *k_out;        // heads
  __nv_bfloat16 *v_out;        // values, or the outputs of a plain product
  long long out_stride;        // elements
  int n_rows, nr;              // rows, and rows rounded up to a multiple of 8
  int row_chunks;              // 16-byte chunks per row
  int n_cols, k_cols;          // columns; those below k_cols are keys
  int tile, n_tiles;           // columns per tile, tiles
  int num_k_blocks, stage_kb;  // k blocks in all and per stage
  int stages, tail_off, tmem_cols;  // shared and tensor memory
  int wide_store;              // plain product: outputs are 32-byte aligned
  float inv_k, rms_eps;
  int qk_norm;
  float qk_eps;
  int rope_half;
  int max_pos;
  const float2 *rope_hi, *rope_lo;
  const float *gamma_k;
  int *status;
  unsigned long long timeout_ns;
  uint4 *append_rows;          // as in RecomputeParams; nullptr: nothing is appended
  int32_t *append_pos;
  float *append_sumsq;
  long long append_slot[RW_MAX_ROWS];
  long long store_slots;       // slots of the store (checking build)
};

// ------------------------------------------------------------------------------ decode attention
constexpr int AT_THREADS = 128;        // streaming kernel
constexpr int AT_WARPS = 4;
constexpr int AT_CTAS_PER_SM = 4;      // 128 registers per thread
constexpr int AT_MERGE_THREADS = 640;  // merge kernel: at most 20 warps (102 registers each)
constexpr int AT_MERGE_WARPS = 20;
constexpr int AT_MERGE_SLICE = 64;     // channels per merge CTA
constexpr int AT_TAIL_KEYS = 8;        // live keys per sequence that the merge kernel takes itself, behind a fused recompute
// partials one warp of the merge kernel fetches at once: 4*G registers each, 64 registers in all
constexpr int attn_merge_group(int g) { return 16 / g >= 1 ? 16 / g : 1; }
constexpr int AT_UNROLL = 8;          // keys per lane group per iteration
constexpr int AT_MAX_SEQS = 64;       // sequences per launch (bounded by the kernel parameter space)

struct AttnSeq {
  const __nv_bfloat16 *k[KVD_MAX_SEGMENTS];
  const __nv_bfloat16 *v[KVD_MAX_SEGMENTS];
  long long stride[KVD_MAX_SEGMENTS];
  int first[KVD_MAX_SEGMENTS];
  int len[KVD_MAX_SEGMENTS];
  int q_pos;
  int lo_pos;       // first visible position
  int hi_pos;       // last visible position (<= q_pos)
  int chunk0_pos;   // position of the first key of chunk 0 (multiple of the chunk size)
  int n_chunks;
  int part_base;    // chunks of the sequences before this one in the launch (the flattened grid)
  int iters;        // warp iterations per chunk
  int slot_base;    // slot of this sequence's chunk 0 in the partial arrays
  int merge_base;   // first slot and number of slots the merge kernel combines for this sequence: the
  int merge_count;  // streaming kernel's chunks, preceded by partials of the fused recompute kernel if any
};

// Live keys that the merge kernel attends itself: visible, and not cut into chunks.
__host__ __device__ inline bool attn_tail(const AttnSeq &S) { return S.n_chunks == 0 && S.hi_pos >= S.lo_pos; }

// Launch-wide fields, followed by the per-sequence descriptors.  The kernel takes the variant whose
// array is just large enough (AttnLaunchT<4> for small batches: a 10 KB parameter block costs
// microseconds to launch).
struct AttnLaunchHead {
  int n_seqs;
  int total_chunks;
  int n_q;
  int n_kv;
  float scale_log2e;
  const __nv_bfloat16 *q;  // [n_seqs, n_q, d_head] (already offset to the launch's first sequence)
  __nv_bfloat16 *out;      // [n_seqs, n_q, d_head]
  float *part_o;           // [parts][n_q][d_head]
  float *part_ml;          // [parts][n_q][2]
  int *status;             // device status word (nullptr: none), used by the checking build
  int max_parts;           // slots the partial arrays hold
  bool early;              // both kernels start early whatever their grids
  bool tail;               // there is a sequence whose live keys the merge kernel attends itself (attn_tail)
};
template <int NSEQ>
struct AttnLaunchT : AttnLaunchHead {
  AttnSeq seq[NSEQ];
};
typedef AttnLaunchT<AT_MAX_SEQS> AttnLaunch;

// keys per chunk for a head size and iteration count
inline int attn_keys_per_warp_iter(int d_head) { return (32 / (d_head / 8)) * AT_UNROLL; }
// Iterations per chunk.  Spans up to 8192 keys are cut into at most 128 chunks per (sequence, KV
// head), longer ones so that one sequence yields about 592 work units (chunks x KV heads) -- four
// CTAs on each of a B200's 148 SMs -- which keeps every SM equally loaded when the batch is 1.  A
// chunk is at least two iterations: a CTA's prologue and combine cost as much as streaming a few
// dozen keys, and in batched launches one-iteration CTAs measured 20 % slower.  A function of the
// model and of the visible span only, so a full cache and a recomputed + window + current layout
// of the same positions are split identically, and a sequence's result does not depend on what
// else is in the batch.
inline int attn_target_chunks(int n_kv, int span) {
  if (span <= 8192) return 128;
  const int t = (148 * AT_CTAS_PER_SM) / n_kv;
  return t > 16 ? t : 16;
}
inline int attn_iters_for_span(int d_head, int n_kv, int span) {
  const int per_iter = attn_keys_per_warp_iter(d_head) * AT_WARPS;
  const long long per_chunk_min = static_cast<long long>(per_iter) * attn_target_chunks(n_kv, span);
  long long iters = (span + per_chunk_min - 1) / per_chunk_min;
  if (iters < 2) iters = 2;
  if (iters > 64) iters = 64;
  return static_cast<int>(iters);
}
inline int attn_chunk_keys(int d_head, int iters) { return attn_keys_per_warp_iter(d_head) * AT_WARPS * iters; }
inline int attn_max_chunks(int d_head, int n_kv, int max_tokens) {
  const int per_iter = attn_keys_per_warp_iter(d_head) * AT_WARPS;
  const int capped = max_tokens / (per_iter * 64) + 2;  // once the iteration count is capped
  int target = attn_target_chunks(n_kv, max_tokens);
  if (target < 128) target = 128;
  return (capped > target ? capped : target) + 2;
}

// ------------------------------------------------------------------------------ context
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct RopeTable {
  float2 *hi = nullptr;
  float2 *lo = nullptr;
  int n_hi = 0;
};

struct LayerState {
  bool set = false;
  __nv_bfloat16 *wt = nullptr;  // [2*n_kv*d_head, d_hidden]: gamma-folded, K-major
  float *gamma_k = nullptr;     // [d_head] fp32
  float theta = 0.f;
  int window = 0;
  RopeTable rope;
  CUtensorMap tmap_b;
  CUtensorMap tmap_b_part[2];  // the same with boxes of a half and of a quarter of a tile's columns
  CUtensorMap tmap_rows[2];  // of wt, for the projection of few and of more rows (16-bit types), and its columns per tile
  int rows_tile = 0;
  // FP8 variant: E4M3 codes of W' / w_scale8, K-major; one scale for the matrix (device float)
  uint8_t *wt8 = nullptr;
  float *w_scale8 = nullptr;
  CUtensorMap tmap_b8;
};

}  // namespace kvd

struct kvd_ctx {
  kvd_model_desc desc;
  int device = 0;
  int num_sms = 0;
  int block_n = 0;
  int dtype = 0;  // 16-bit element type of rows, weights and K/V: 0 bf16, 1 fp16 (recompute path only)
  std::vector<kvd::LayerState> layers;
  std::map<uint32_t, kvd::RopeTable> rope_cache;  // keyed by the bits of theta
  // residual store
  __nv_bfloat16 *store_rows = nullptr;
  int32_t *store_pos = nullptr;
  float *store_sumsq = nullptr;
  float *ext_sumsq = nullptr;     // statistics of caller rows taken ahead of the recompute kernel
  size_t ext_sumsq_rows = 0;
  unsigned long long *argmax_keys = nullptr;  // scaffold greedy pick: one slot per row
  size_t argmax_rows = 0;
  int32_t *zero_pos = nullptr;    // ext_sumsq_rows zeros: the positions of rows that are not rotated (scaffold products)
  int layers_stored = 0;
  std::vector<int> rows_stored;  // [layers_stored * max_seqs]
  std::vector<CUtensorMap> store_maps;  // per stored layer: [max_seqs][max_tokens_per_seq][d_hidden]
  // FP8 residual store (separate arena): codes, positions, sums of squares of the original rows, scales
  uint8_t *store8_codes = nullptr;
  int32_t *store8_pos = nullptr;
  float *store8_sumsq = nullptr;
  float *store8_scale = nullptr;
  int layers_stored8 = 0;
  std::vector<int> rows_stored8;
  std::vector<CUtensorMap> store8_maps;
  // FP4 residual store (a third arena): E2M1 codes, E4M3 block scales, positions, sums of squares, row scales
  uint8_t *store4_codes = nullptr;
  uint8_t *store4_block = nullptr;
  int32_t *store4_pos = nullptr;
  float *store4_sumsq = nullptr;
  float *store4_scale = nullptr;
  int layers_stored4 = 0;
  std::vector<int> rows_stored4;
  unsigned *amax_scratch = nullptr;  // one word, used while weights are prepared
  // attention scratch
  float *part_o = nullptr;
  float *part_ml = nullptr;
  size_t workspace_bytes = 0;
  int max_parts = 0;
  int *d_status = nullptr;
  uint64_t launches = 0;
  uint64_t prepared_bytes = 0;
  unsigned long long timeout_ns = 2000000000ull;
  long long *trace = nullptr;
  size_t trace_bytes = 0;
  kvd::LaunchMark few_rows;  // the last launch of the few-row kernel that made keys and values
  std::string last_error;
  kvd::EncodeTiledFn encode = nullptr;
};

namespace kvd {
// Kernels are launched as programmatic dependents of their predecessor in the stream unless the
// environment variable KVD_SERIAL_LAUNCH says otherwise: a bit mask, 1 = recompute and few-row kernels, 2 = attention
// streaming kernel, 4 = attention merge kernel, 8 = all others get plain stream ordering instead.
inline int serial_launch_mask() {
  static const int mask = [] {
    const char *e = getenv("KVD_SERIAL_LAUNCH");
    return e ? atoi(e) : 0;
  }();
  return mask;
}

// A kernel launched as a programmatic dependent runs while its predecessor does.  What the predecessor may still write
// (rows, positions, statistics, codes) it therefore reads by plain loads behind grid_dependency_wait(): no __ldg (the
// non-coherent load is for memory that nobody writes during the kernel), and, in the kernels started by the function
// below, no __restrict__ on an argument (it permits a load to move above the wait).  __ldg is for tables and weights,
// which are complete before the first launch that reads them.  (Keys, values and queries as well: decode attention's
// streaming loads cost the same without the non-coherent path, 32768 cached keys 36.7 us per step either way, 16 x 2048
// 38.6.)
//
// Launch of a small kernel that calls grid_dependency_wait() before it touches memory: as a programmatic dependent of
// its predecessor, so that its launch latency and the predecessor's end overlap (three decoder blocks at batch 1, 35
// launches: 459 -> 421 us) -- if its grid leaves half of the SMs free.  Larger grids are ordered plainly: the next
// kernel's CTAs then wait on SMs this one still needs (decoding 3000 FP4 rows ahead of their projection: 56 -> 66 us
// for the step with an early start).
template <typename... P, typename... A>
inline cudaError_t launch_dependent(const kvd_ctx *ctx, void (*kern)(P...), dim3 grid, unsigned threads, cudaStream_t stream, A &&...args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = (serial_launch_mask() & 8) || 2 * grid.x > static_cast<unsigned>(ctx->num_sms) ? 0 : 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Schedule of a launch: its tiles (units of two, single ones, cut ones) and its CTA pairs.  The one place both the launch
// and the size test of the trace buffer take the grid from.
struct RcSchedule {
  int unit_tiles, whole_tiles, parts, clusters;
};
RcSchedule rc_schedule(int num_sms, int block_n, int d_head, int m_blocks, int n_blocks, int k_blocks, int k_cols, int eb, bool fused);
inline size_t rc_trace_bytes(int clusters) {
  return 2 * static_cast<size_t>(clusters) * RC_TRACE_TILES * RC_TRACE_FIELDS * sizeof(long long);
}
// After the sizes of `p` are known: its schedule, and the trace buffer if the launch fits it.
inline void schedule_recompute(const kvd_ctx *ctx, RecomputeParams &p, int eb, bool fused) {
  const RcSchedule s = rc_schedule(ctx->num_sms, ctx->block_n, ctx->desc.d_head, p.num_m_blocks, p.num_n_blocks, p.num_k_blocks, p.k_cols, eb, fused);
  p.unit_tiles = s.unit_tiles;
  p.whole_tiles = s.whole_tiles;
  p.parts = s.parts;
  p.clusters = s.clusters;
  // (fp16 and fp32 kernels record nothing, and the hook must not choose the kernel of a call it cannot trace)
  p.trace = ctx->trace && ctx->dtype == KVD_DTYPE_BF16 && rc_trace_bytes(s.clusters) <= ctx->trace_bytes ? ctx->trace : nullptr;
}
// launchers implemented next to their kernels
kvd_status launch_recompute(kvd_ctx *ctx, const LayerState &ls, const CUtensorMap &tmap_store,
                            const CUtensorMap &tmap_rows, const RecomputeParams &p, cudaStream_t stream);
kvd_status launch_recompute_fused(kvd_ctx *ctx, const LayerState &ls, const CUtensorMap &tmap_store,
                                  const CUtensorMap &tmap_rows, const RecomputeParams &p, const FusedParams &fp,
                                  cudaStream_t stream, int eb = 2);
// `heads`: key and value heads of a layer; otherwise a plain product (bf16)
kvd_status prepare_rows_map(kvd_ctx *ctx, LayerState &ls, int k, int n_cols, bool heads);
kvd_status launch_rows(kvd_ctx *ctx, const LayerState &ls, int k, RowsParams &p, bool heads, cudaStream_t stream);
kvd_status launch_attention(kvd_ctx *ctx, const AttnLaunch &L, int d_head, int group, cudaStream_t stream);
kvd_status launch_prepare_weights(kvd_ctx *ctx, const __nv_bfloat16 *w, const __nv_bfloat16 *gamma, __nv_bfloat16 *wt,
                                  int d_hidden, int n_cols, cudaStream_t stream);
kvd_status launch_convert_gamma(kvd_ctx *ctx, const __nv_bfloat16 *g, float *out, int n, cudaStream_t stream);
kvd_status launch_rowstats(kvd_ctx *ctx, const __nv_bfloat16 *rows, float *sumsq, int n, int d_hidden,
                           cudaStream_t stream);
kvd_status launch_checkpoint_fp8(kvd_ctx *ctx, const __nv_bfloat16 *rows, const int32_t *pos, uint8_t *dst_codes,
                                 int32_t *dst_pos, float *dst_sumsq, float *dst_scale, int n, int d_hidden,
                                 cudaStream_t stream);
kvd_status launch_prepare_weights_fp8(kvd_ctx *ctx, const __nv_bfloat16 *w, const __nv_bfloat16 *gamma, uint8_t *wt8,
                                      int d_hidden, int n_cols, unsigned *amax_scratch, float *scale_out,
                                      cudaStream_t stream);
kvd_status launch_recompute_fp8(kvd_ctx *ctx, const LayerState &ls, const CUtensorMap &tmap_store,
                                const CUtensorMap &tmap_rows, const RecomputeParams &p, cudaStream_t stream);
kvd_status launch_checkpoint(kvd_ctx *ctx, const __nv_bfloat16 *rows, const int32_t *pos, __nv_bfloat16 *dst_rows,
                             int32_t *dst_pos, float *dst_sumsq, int n, int d_hidden, cudaStream_t stream);
kvd_status launch_selftest_bounds(kvd_ctx *ctx, cudaStream_t stream);
kvd_status launch_checkpoint_scatter(kvd_ctx *ctx, const __nv_bfloat16 *rows, const int32_t *pos, const CkptSlots &slots,
                                     int n, int d_hidden, cudaStream_t stream);
// kvd_prefill_attention: many query tokens of one sequence, tiled over query rows (Eq. 6-7 per row)
struct PrefillParams {
  const __nv_bfloat16 *q;    // [n_rows][n_q][d_head]
  __nv_bfloat16 *out;        // [n_rows][n_q][d_head]
  const int32_t *q_pos;      // DEVICE [n_rows]
  int n_rows, n_q, n_kv, window;
  float scale_log2e;
  int seg_lo, seg_hi;        // first and last position any segment holds
  const __nv_bfloat16 *k[KVD_MAX_SEGMENTS];
  const __nv_bfloat16 *v[KVD_MAX_SEGMENTS];
  long long stride[KVD_MAX_SEGMENTS];
  int first[KVD_MAX_SEGMENTS];
  int len[KVD_MAX_SEGMENTS];
  int *status;                    // device status word
  unsigned long long timeout_ns;  // limit of every in-kernel wait
};
// the tcgen05 form of the call (128 MMA rows per CTA, scores and outputs in tensor memory)
kvd_status launch_prefill_tc(kvd_ctx *ctx, const PrefillParams &P, int d_head, int group, cudaStream_t stream);
kvd_status launch_selftest_timeout(kvd_ctx *ctx, unsigned long long timeout_ns, cudaStream_t stream);
kvd_status cuda_fail(kvd_ctx *ctx, cudaError_t e, const char *where);
// host helpers shared by the entry points (kvd_api.cu)
kvd_status encode_2d(kvd_ctx *ctx, CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer,
                     uint32_t box_inner, uint32_t box_outer, int eb = 2);
kvd_status encode_rows_3d(kvd_ctx *ctx, CUtensorMap *map, const void *base, uint64_t d_hidden, uint64_t rows,
                          uint64_t slabs, int eb = 2);
kvd_status get_rope(kvd_ctx *ctx, float theta, RopeTable *out);
}  // namespace kvd
