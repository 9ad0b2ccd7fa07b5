// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "seer.h"

namespace seer {

constexpr int kBlock = 64;      // attention tile; the gate block is 64 or 128 tokens (SeqMeta::block)
constexpr int kHeadDim = 128;
constexpr int kGateDim = 128;
constexpr int kMaxBatch = 4096;
constexpr int kMetaSlots = 8;
constexpr int kPairWords = 63;  // words of the answer whether pairs of query blocks share their lists (attn_pair.cu)
constexpr int kScoreTile = 64;  // column tile of the gate's score kernel, and granularity of the bands of the one-call gate + mask

// Per-batch metadata the kernels read from device memory.
struct SeqMeta {
  const int32_t* cu_seqlens;   // [batch+1] token offsets
  const int32_t* blk_off;      // [batch+1] cumulative number of blocks
  const int64_t* score_off;    // [batch+1] Hq * cumulative nb^2
  int32_t batch;
  int32_t num_q_heads;
  int32_t num_kv_heads;
  int32_t group;               // Hq / Hkv
  int32_t total_tokens;
  int32_t total_blocks;
  int32_t max_nb;
  int64_t rows;                // Hq * total_blocks
  int64_t score_elems;
  float softmax_scale;
  int32_t block;               // tokens per gate block: 64, or 128 (gate and mask only)
  // chunked prefill (all zero without a chunk): the queries of sequence b are its last positions
  const int32_t* qoff;         // [batch] block position of the chunk's first query block
  const int32_t* qdelta;       // [batch] token index in q / o / lse = token index in k / v + qdelta
  // the attention's order of the sequences
  const int4* place;           // [batch] (first token, tokens, first block, qdelta) of the sequence at each place
  const int32_t* qblk_off;     // [batch + 1] blocks with queries at the places before
  const int32_t* pair_off;     // [batch + 1] pairs of blocks (2u, 2u + 1) with queries at the places before
  int64_t pair_units;          // such pairs, all heads
  int32_t total_q_tokens;      // tokens in q / o / lse
  int32_t chunked;             // 1 if the shape carries cu_seqlens_q
  // bounded waits of the tcgen05 attention kernel, and the test hook that makes one of them run out
  uint32_t wait_limit_us;      // a barrier wait that lasts this long is declared lost
  int64_t score_tiles;         // host: 128 x 64 tiles of the score matrix, all heads, about
  int64_t q_rows;              // host: rows that have queries (all of them without a chunk)
  int32_t first_q_block;       // host: first block of the batch that can have queries (one chunked sequence: where its chunk starts)
  int32_t lose_v_copy;         // >= 0: stream 0 of CTA 0 never issues the V copy of its tile with this ordinal
};

// Projected pooled vectors: per (head, block) three bf16 planes (hi, mid, lo of the fp32 value) of 128 elements.  A head's
// blocks are stored as tiles of 64 (aligned in the packed batch; the last one may be shorter) in the layout the score
// kernel's MMAs read: plane -> k half (64 elements = 128 bytes) -> block of the tile -> 16-byte chunk XOR (block % 8), so that
// a whole tile is one contiguous 48 KB copy.
constexpr int kGatePairBytes = 3 * kGateDim * 2;
struct GateTile {
  size_t base;                 // byte offset from the head's first tile
  int rows;
  __host__ __device__ GateTile(int tile, int total_blocks) : base((size_t)tile * 64 * kGatePairBytes), rows(total_blocks - tile * 64 < 64 ? total_blocks - tile * 64 : 64) {}
};

// Softmax statistics of the gate are formed per segment of this many column tiles (of the packed batch) and combined in order.
__host__ __device__ inline int gate_seg_tiles(int max_nb) { return max_nb <= 2048 ? 4 : 16; }
// segments a sequence of max_nb blocks can touch, wherever it starts
__host__ __device__ inline int gate_stat_segs(int max_nb) { const int c = gate_seg_tiles(max_nb) * kScoreTile; return (max_nb + c - 1) / c + 1; }

// A rectangle of (block row of the packed batch, query head) pairs whose scores are produced and consumed together.
// head_stride == 0: the band's scores lie at (offset in the full score matrix - score_base) in whatever buffer the kernels are
// given.  Otherwise the band is query blocks >= row0 of one sequence, packed: row i of head h lies at
// (h - head_lo) * head_stride + packed_rows(i) - packed_rows(row0), its causal columns alone, rounded up to 64.  A band buffer
// takes twice the heads of whole rows then, and there are as many times fewer launches (32 heads of 4096 blocks in 128 MB: 11 bands
// instead of 32, gate + mask 13 % faster).
struct ScoreBand {
  int32_t blk_lo, blk_hi;      // block rows [blk_lo, blk_hi), numbered over the batch (blk_off)
  int32_t head_lo, heads;
  int64_t score_base;
  int64_t head_stride;
  int32_t row0;
};

// Elements of the packed rows before row i: rows 64 t .. 64 t + 63 take 64 (t + 1) each.
__host__ __device__ inline int64_t packed_rows(int i) {
  const int64_t t = i / kScoreTile, w = kScoreTile;
  return w * w * (t * (t + 1) / 2) + (i - t * w) * w * (t + 1);
}

// Offset of entry (h, i, 0) of sequence b, which has nb blocks.
__device__ __forceinline__ int64_t score_row_offset(const SeqMeta& m, const ScoreBand& sb, int b, int nb, int h, int i) {
  if (sb.head_stride != 0) return (int64_t)(h - sb.head_lo) * sb.head_stride + packed_rows(i) - packed_rows(sb.row0);
  return m.score_off[b] + ((int64_t)h * nb + i) * nb - sb.score_base;
}

struct MetaSlot {
  std::vector<int32_t> key;    // cu_seqlens + Hq: what the slot currently describes
  void* dev = nullptr;
  size_t stage_lo = 0, stage_hi = 0;   // where the staging ring holds what was uploaded last
  cudaEvent_t ready = nullptr;     // upload finished
  cudaEvent_t last_use = nullptr;  // last library call that read the slot
  uint64_t stamp = 0;
};

}  // namespace seer

struct seer_ctx {
  int device = 0;
  int num_sms = 0;
  int* d_status = nullptr;
  int attn_impl = 0;
  int64_t launches = 0;
  uint64_t clock = 0;
  seer::MetaSlot slots[seer::kMetaSlots];
  void* stage = nullptr;           // page-locked ring the slots' uploads start from
  size_t stage_pos = 0;
  void* tmap_encode = nullptr;   // cuTensorMapEncodeTiled, resolved at run time
  void* trace = nullptr;         // optional device buffer for the attention kernel's timeline (diagnostics)
  bool pair_kernels = false;     // their shared-memory limits are set (by the first call that may use them: 0.1 ms of creating a context)
  uint32_t wait_limit_us = 2000000u;   // seer_debug_lost_wait
  int32_t lose_v_copy = -1;
  // seer_prefill_host: copy streams and the events of its two-deep pipeline over KV-head slices
  cudaStream_t h2d_stream = nullptr, d2h_stream = nullptr;
  cudaEvent_t ev_start = nullptr, ev_h2d[2] = {nullptr, nullptr}, ev_comp[2] = {nullptr, nullptr},
              ev_d2h[2] = {nullptr, nullptr};
};

namespace seer {

// Validates the shape, makes its metadata resident on the device (ordered before later work on `stream`)
// and fills `m`.  `slot_out` identifies the slot to pass to finish_call.  `keep`: a slot that the same call has prepared before, which
// is not taken for this shape though nothing in flight reads it yet.
seer_status prepare(seer_ctx* ctx, const seer_shape* shape, cudaStream_t stream, SeqMeta* m, int* slot_out, int keep = -1);
void finish_call(seer_ctx* ctx, int slot, cudaStream_t stream);
// Whether tensors that the kernels copy 16 bytes at a time begin on 16 bytes (a misaligned access would end the context).
bool on_16(const void* a, const void* b, const void* c = nullptr, const void* d = nullptr);

// Host-only shape arithmetic (no CUDA calls): returns SEER_OK and fills totals.
struct ShapeTotals {
  int64_t total_tokens, total_q_tokens, total_blocks, rows, score_elems, causal_blocks;
  int32_t max_nb;
};
seer_status shape_totals(const seer_shape* shape, ShapeTotals* t);

size_t gate_workspace_bytes(const ShapeTotals& t, const seer_shape* shape);   // the projected vectors
size_t gate_stats_bytes(const ShapeTotals& t, const seer_shape* shape);       // the softmax statistics that may follow them

// The gate's row softmax, everything in units of log2: x = logit * log2(e), m the maximum of x, l the sum of 2^(x - m).
__device__ __forceinline__ float gate_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gate_score(float x, float row_m, float inv_l) { return __fmul_rn(gate_ex2(__fsub_rn(x, row_m)), inv_l); }
// (m, l) of two disjoint sets of a row's columns; m = -inf: empty
__device__ __forceinline__ void gate_combine(float& m, float& l, float m2, float l2) {
  const float inf = __int_as_float(0x7f800000), nm = fmaxf(m, m2);
  const float f = m == -inf ? 0.f : gate_ex2(m - nm), f2 = m2 == -inf ? 0.f : gate_ex2(m2 - nm);
  l = __fadd_rn(__fmul_rn(l, f), __fmul_rn(l2, f2));
  m = nm;
}
// Statistics of block row gb (numbered over the batch) of head h, whose sequence starts at block `start`.
__device__ __forceinline__ void gate_row_stats(const SeqMeta& m, const float2* stats, int h, int gb, int start, float& row_m, float& row_l) {
  const int seg_cols = gate_seg_tiles(m.max_nb) * kScoreTile, segs = gb / seg_cols - start / seg_cols + 1;
  const float2* st = stats + ((size_t)h * m.total_blocks + gb) * gate_stat_segs(m.max_nb);
  row_m = __int_as_float(0xff800000); row_l = 0.f;
  for (int s = 0; s < segs; ++s) { const float2 v = st[s]; gate_combine(row_m, row_l, v.x, v.y); }
}

// Launch of a kernel that may start while its predecessor in the stream still runs (programmatic dependent launch): its CTAs get
// ready as the predecessor's leave, and grid_wait() in the kernel holds them until the predecessor has completed and its writes are
// visible.  Every CTA calls it, on every path, before it touches anything but its arguments and the shape's offsets (uploaded
// before the call's first kernel): a grid that ended without it would let its successor overtake its predecessor.  Only
// then does a kernel let its own successor start: two kernels overlap, never three, so no line that a third one rewrites can
// sit in L1, and a kernel that rewrites what it has read reads past L1.
// It is worth the start of a kernel, about 2 us, at each of a call's launches: 2k tokens, four heads, 48.5 us without and 36.2 with it.
template <typename... P, typename... A>
cudaError_t launch_next(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// What the kernel before writes (scores, statistics, projected vectors, row_ptr, col_idx, lse) changes while this kernel is resident,
// so nothing may promise the compiler that it does not: no __restrict__ and no __ldg on it, which allow a load to move above the
// wait.  These loads name the address space of a pointer that the compiler has lost sight of.
__device__ __forceinline__ uint32_t ld_global(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_global_v4(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// Kernel launchers (each returns the number of kernels it launched, or a negative cudaError).
int launch_gate(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const float* Wq, const float* Wk,
                float* scores, void* ws, size_t ws_bytes, cudaStream_t stream);
int launch_gate_ex(seer_ctx* ctx, const SeqMeta& m, const seer_gate_options& opt, const void* q, const void* k,
                   const float* Wq, const float* Wk, float* scores, void* ws, size_t ws_bytes, cudaStream_t stream);
// The one-call gate + mask: statistics of all rows once, then the scores of one band at a time, from the vectors a launch with
// scores == nullptr left in `ws`.
int launch_gate_stats_all(seer_ctx* ctx, const SeqMeta& m, void* ws, cudaStream_t stream);
int launch_gate_scores_band(seer_ctx* ctx, const SeqMeta& m, const ScoreBand& band, void* ws, float* scores, bool with_stats,
                            cudaStream_t stream);
// ... or its logits (units of log2) and its rows' statistics at once, for launch_mask_band with `logits`.
int launch_gate_logits_band(seer_ctx* ctx, const SeqMeta& m, const ScoreBand& band, void* ws, float* logits, cudaStream_t stream);
const float2* gate_stats(const SeqMeta& m, void* ws);
bool gate_logits_pay(const SeqMeta& m, int64_t bands, int num_sms);   // bands of logits, or statistics and bands of scores?
bool gate_split(const SeqMeta& m, int num_sms);   // scores of the whole problem: statistics apart from the scores?
// Mask rows [row_lo, row_hi) from a band of scores; `first` starts row_ptr at 0, later bands continue from the
// previous band's last entry; `stats` (or nullptr) are the statistics the scores were made from; `logits`: `scores` holds logits
// (mask_takes_logits).
bool mask_takes_logits(const SeqMeta& m, const seer_mask_params& p);
int launch_mask_band(seer_ctx* ctx, const SeqMeta& m, const float* scores, const float2* stats, bool logits, const ScoreBand& sb, int64_t row_lo,
                     int64_t row_hi, bool first, const seer_mask_params& p, int32_t* row_ptr, int32_t* col_idx,
                     int64_t col_capacity, int64_t* nnz_out, cudaStream_t stream);
// 128-token block lists -> the 64-token lists the attention kernels take (m128 and m64 describe the same batch).
int launch_expand_lists(seer_ctx* ctx, const SeqMeta& m128, const SeqMeta& m64, const int32_t* row_ptr128,
                        const int32_t* col_idx128, int32_t* row_ptr64, int32_t* col_idx64, int64_t col_capacity64,
                        int64_t* nnz_out, cudaStream_t stream);
int launch_mask(seer_ctx* ctx, const SeqMeta& m, const float* scores, const seer_mask_params& p, int32_t* row_ptr,
                int32_t* col_idx, int64_t col_capacity, int64_t* nnz_out, cudaStream_t stream);
int launch_attn_mma(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const void* v,
                    const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, cudaStream_t stream);
int launch_block_max(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const int32_t* row_ptr,
                     const int32_t* col_idx, const float* lse, float* out, cudaStream_t stream);
int launch_block_max_tc(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const int32_t* row_ptr,
                        const int32_t* col_idx, const float* lse, float* out, cudaStream_t stream);
int launch_attn_tc(seer_ctx* ctx, const SeqMeta& m, const void* q, const void* k, const void* v,
                   const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, int* work_counter,
                   cudaStream_t stream);
seer_status init_gate(seer_ctx* ctx);
seer_status init_mask(seer_ctx* ctx);
seer_status init_attn_mma(seer_ctx* ctx);
seer_status init_attn_tc(seer_ctx* ctx);


// Sequence that owns global block index gb: largest b with blk_off[b] <= gb (empty sequences are skipped).
__device__ __forceinline__ int find_sequence(const int32_t* __restrict__ off, int batch, int x) {
  int lo = 0, hi = batch;  // off[lo] <= x < off[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (off[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

}  // namespace seer
