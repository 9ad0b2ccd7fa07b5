// AttnGate, second stage (Sec. 3.1, Eq. 1): logits = gq gk^T / sqrt(dg) over the causal blocks, row softmax -> scores.
//
// The logits need fp32-grade products (bf16 or tf32 inputs would not hold the 1e-3 relative bound on softmax outputs
// when logits reach tens), so gq and gk arrive as three bf16 planes each, x = hi + mid + lo, and the product is the six
// terms hi*lo + lo*hi + mid*mid (small) and hi*mid + mid*hi + hi*hi (large) (what is dropped is below 2^-24 of the
// product), accumulated in fp32 TMEM accumulators by tcgen05.mma: 6 x 8 K-steps of M = 128, N = 64, K = 16 per tile.
//
// What bounds it: the MMAs.  The rows' planes are the A operand in tensor memory (192 columns, written once per CTA):
// an MMA then reads 2 KB of shared memory instead of 6 and takes 34 clocks instead of 48.
//
// One CTA = 128 consecutive block rows of one head (rows of the packed batch, whatever sequences they belong to) times a
// range of column tiles of 64 blocks (tiles of the packed batch, aligned to 64).  A score needs the softmax statistics of
// its whole row first, so every tile is computed twice (unless there are two at most) and every score is written once:
//   kBoth   one CTA walks all causal tiles of its rows twice (short sequences: one launch)
//   kStats  a CTA walks one segment of up to SegTiles tiles and leaves the rows' (maximum, sum) of that segment
//   kWrite  a CTA walks part_tiles tiles, after combining its rows' statistics, and writes exp(x - m) / l
// Where the scores are only read again by this library's selection, which can form them itself, one sweep is enough:
//   kLogits a CTA walks part_tiles tiles, whole segments, and leaves the logits and the segments' statistics
// (lists of 262 144 tokens, 32 heads: 2.40 ms by statistics of all rows, then scores band by band; 2.11 so; 8k tokens against 128k:
// 163 and 142 us; 917 against 60k in a batch of four: 90 and 74).
// With long sequences the first form has few CTAs of very unequal length (one head of a 262 144-token prompt: 32 CTAs, 245 us
// a launch).  Statistics are always formed per segment of the batch's column grid and combined in segment order, so the
// scores are the same bit for bit whichever form computes them and however the rows are grouped into calls.
//
// Roles (608 threads): warps 0-15 own the rows in two groups, one for the even, one for the odd tiles of the column grid, each
// with an accumulator pair of its own (a warp takes 32 rows x 32 of a tile's 64 columns: TMEM lane = row, so maxima and sums
// need no shuffle; one group took 2900 clocks per tile, the MMAs 1650); one thread of warp 16 issues the small terms, one of
// warp 17 the large ones, each into its own accumulator (the rows add the two), one of warp 18 copies the column tiles (one
// 48 KB bulk copy each: the first stage stores the planes in the swizzled tile layout).  A finished tile goes through shared
// memory so that a warp writes whole 128-byte row segments (a thread storing its own row scatters 16-byte pieces over 32 rows:
// three times slower).
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>

#include "attn_tc_common.cuh"
#include "seer_internal.cuh"

namespace seer {

using namespace tcc;

namespace gs {
constexpr int kRows = 128;                         // score rows per CTA
constexpr int kCols = kScoreTile;                  // columns per tile (64)
constexpr int kRowThreads = 512;                   // two groups of eight warps
constexpr int kThreads = kRowThreads + 96;
constexpr uint32_t kBPlane = kCols * kGateDim * 2;   // 16 KB: one plane of a column tile, [2 k halves][64 rows][128 B]
constexpr uint32_t kBBuf = 3 * kBPlane;
constexpr uint32_t kBBufs = 3;
constexpr uint32_t kOffStage = kBBufs * kBBuf;       // 16 warps x [32 rows][32 columns] fp32
constexpr uint32_t kOffSeg = kOffStage + 16 * 4096;    // (m, l) of a segment: [segment parity][group][half][row]
constexpr uint32_t kOffMeta = kOffSeg + 8 * kRows * 8;   // per row: element offset of column 0 (int64), first and last causal block
constexpr uint32_t kOffBar = kOffMeta + kRows * 16;
constexpr uint32_t kOffMisc = kOffBar + 128;         // tmem base, abort flag
constexpr uint32_t kSmemBytes = kOffMisc + 64;
static_assert(kSmemBytes <= 232448, "shared memory budget of one CTA");
enum Bar { ACC_FULL = 0 /* + acc */, ACC_EMPTY = 2, B_FULL = 4 /* + buf */, B_EMPTY = 4 + kBBufs, A_FULL = 4 + 2 * kBBufs, kBars = A_FULL + 1 };
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColA = 256;                      // columns 0..255: two accumulator pairs; 256..447: the A planes
constexpr uint32_t kIdesc = make_idesc(false, false, kCols);
constexpr uint32_t kWaitSpins = 1u << 24;            // a wait that lasts this many polls (seconds) is declared lost
enum Mode { kBoth = 0, kStats = 1, kWrite = 2, kLogits = 3 };

// Bounded wait that never changes the control flow: after the limit the error is recorded and the wait counts as
// satisfied, so every role still reaches its barriers and the CTA ends normally (with a wrong result and a status).
__device__ __forceinline__ void wait_bar(uint32_t bar, uint32_t parity, uint32_t abort_addr, int* status) {
  for (uint32_t it = 0; it < kWaitSpins; ++it) {
    if (mbar_try(bar, parity)) return;
    if ((it & 255u) == 255u && ld_shared_u32(abort_addr) != 0u) return;
  }
  st_shared_u32(abort_addr, 1u);
  if (status != nullptr) atomicCAS(status, 0, (int)SEER_ERR_TIMEOUT);
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Parts of a row tile's causal columns when the batch is one sequence.
__host__ __device__ __forceinline__ int part_count(const ScoreBand& band, int tile, int part_tiles) {
  const int r0 = band.blk_lo + tile * kRows, last = (band.blk_hi - r0 < kRows ? band.blk_hi - r0 : kRows) + r0 - 1;
  return last / (part_tiles * kCols) + 1;
}

}  // namespace gs

// grid.x = row tiles * band.heads (head fastest; row tiles are visited from the last rows to the first), grid.y = parts of
// part_tiles column tiles (part_tiles = 0, always so for kBoth: one part; for kStats a part is a segment); with one sequence in the batch the parts are in grid.x
// (a CTA that has nothing to do still takes an SM to itself for 2 us).  Row r of a tile is query block i_r of sequence b_r; its causal columns are the blocks seq_start_r .. r of
// the batch.  The whole problem is the band (0, total_blocks, 0, Hq, 0).  Scores are written at their offset in the full
// matrix minus band.score_base.  stats: [head][block of the batch][stat_segs] (m, l).
template <int kMode>
__global__ void __launch_bounds__(gs::kThreads, 1)
gate_scores_kernel(SeqMeta m, ScoreBand band, const uint16_t* gq, const uint16_t* gk,
                   float* scores, float2* stats, int* __restrict__ status, int part_tiles) {
  using namespace gs;
  extern __shared__ __align__(1024) unsigned char gs_raw[];   // (the swizzled tiles need 1024-byte alignment)
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(gs_raw);
  unsigned char* smem = gs_raw;
  if ((base & 1023u) != 0u) {
    grid_wait();
    if (threadIdx.x == 0 && status != nullptr) atomicCAS(status, 0, (int)SEER_ERR_CUDA);
    return;
  }
  const uint32_t bar0 = base + kOffBar, abort_addr = base + kOffMisc + 4;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  const int row_tiles = (band.blk_hi - band.blk_lo + kRows - 1) / kRows;
  int tile = row_tiles - 1 - (int)(blockIdx.x / band.heads), part_of_tile = (int)blockIdx.y;
  const bool parted = kMode != kBoth && part_tiles != 0;
  if (parted && m.batch == 1) {                                   // only the parts that exist: row tile t has part_count of them
    int rest = (int)(blockIdx.x / band.heads);
    for (tile = row_tiles - 1; tile > 0; --tile) {
      const int parts = part_count(band, tile, part_tiles);
      if (rest < parts) break;
      rest -= parts;
    }
    part_of_tile = rest;
  }
  const int h = band.head_lo + (int)(blockIdx.x % band.heads);
  const int g = h / m.group;
  const int r0 = band.blk_lo + tile * kRows;                              // first block row of the tile
  const int rows_valid = min(kRows, band.blk_hi - r0);
  const int seg_cols = gate_seg_tiles(m.max_nb) * kCols;
  const int stat_segs = gate_stat_segs(m.max_nb);

  const int first_col = m.blk_off[find_sequence(m.blk_off, m.batch, r0)]; // rows ascend, so do their sequence starts
  const int last_col = r0 + rows_valid - 1;
  int col_lo = first_col, col_hi = last_col;                              // columns of this CTA
  if (parted) {
    const int part_cols = part_tiles * kCols, part = first_col / part_cols + part_of_tile;
    col_lo = max(col_lo, part * part_cols);
    col_hi = min(col_hi, (part + 1) * part_cols - 1);
    if (col_lo > col_hi) { grid_wait(); return; }
  }

  // this thread's row (threads t, t + 128, .. share row t; the helpers only need the tile's column range)
  const int row = (warp & 3) * 32 + lane;
  int my_start = 0, my_last = -1;
  if (threadIdx.x < kRowThreads && row < rows_valid) {
    const int gb = r0 + row;
    const int b = find_sequence(m.blk_off, m.batch, gb);
    const int nb = m.blk_off[b + 1] - m.blk_off[b];
    const int i = gb - m.blk_off[b];
    my_start = m.blk_off[b];
    if (!(m.chunked && i < m.qoff[b])) my_last = gb;                      // chunked prefill: rows before the chunk are skipped
    if (threadIdx.x < kRows) {
      const long long off = score_row_offset(m, band, b, nb, h, i) - my_start;   // + j = element of column j
      *reinterpret_cast<long long*>(smem + kOffMeta + row * 16) = off;
      *reinterpret_cast<int2*>(smem + kOffMeta + row * 16 + 8) = make_int2(my_start, my_last);
    }
  } else if (threadIdx.x < kRows) {
    *reinterpret_cast<int2*>(smem + kOffMeta + row * 16 + 8) = make_int2(0, -1);
  }
  if (!__syncthreads_or(my_last >= 0 ? 1 : 0)) { grid_wait(); return; }                    // a tile of query blocks before their chunks
  const int tile_lo = col_lo / kCols;
  const int ntiles = col_hi / kCols - tile_lo + 1;                        // column tiles of one sweep
  const int total = kMode == kBoth ? 2 * ntiles : ntiles;
  // of two tiles each group of row warps has one: its logits stay in registers between the sweeps
  const bool kept = kMode == kBoth && ntiles <= 2;
  const int products = kept ? ntiles : total;                             // tiles that are multiplied

  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)kBars; ++i)                                  // one commit per issuing thread; one arrival per row warp
      mbar_init(bar0 + 8 * i, i < ACC_EMPTY ? 2 : i < B_FULL ? 8 : i < (int)B_EMPTY ? 1 : i < (int)A_FULL ? 2 : kRowThreads / 32);
    st_shared_u32(abort_addr, 0u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + kOffMisc), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_wait();
  const uint32_t tmem = *tmem_slot;
  const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
  const int half = (warp >> 2) & 1;                                       // which 32 columns of a tile this row warp takes
  const int grp = (warp >> 3) & 1;                                        // ... and of which tiles: even or odd ones

  // A: the rows' planes, lane = row, two bf16 per column; each of a row's four threads copies a quarter
  if (warp < 16) {
    const int gb = min(r0 + row, m.total_blocks - 1);
    const GateTile at(gb >> 6, m.total_blocks);
    const char* src = reinterpret_cast<const char*>(gq) + (size_t)h * m.total_blocks * kGatePairBytes + at.base + (size_t)half * at.rows * 128 + (size_t)(gb & 63) * 128;
    uint32_t w[3][16];
#pragma unroll
    for (int pl = 0; pl < 3; ++pl)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (my_last >= 0) v = *reinterpret_cast<const uint4*>(src + (size_t)pl * at.rows * 256 + (((grp * 4 + c) ^ (gb & 7)) << 4));
        w[pl][4 * c] = v.x; w[pl][4 * c + 1] = v.y; w[pl][4 * c + 2] = v.z; w[pl][4 * c + 3] = v.w;
      }
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) tc_st16(tmem + lane_addr + kColA + (uint32_t)pl * 64u + (uint32_t)half * 32u + (uint32_t)grp * 16u, w[pl]);
    tc_wait_st();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar0 + 8 * A_FULL);
  }

  if (warp == 18) {
    // ------------------------------------------------------------------------------------------ copies
    if (elect_one()) {
      const char* src = reinterpret_cast<const char*>(gk) + (size_t)g * m.total_blocks * kGatePairBytes;
      uint32_t buf = 0, ph = 1;
      for (int n = 0; n < products; ++n) {
        wait_bar(bar0 + 8 * (B_EMPTY + buf), ph, abort_addr, status);
        const GateTile bt(tile_lo + (n >= ntiles ? n - ntiles : n), m.total_blocks);
        const uint32_t full = bar0 + 8 * (B_FULL + buf), dst = base + buf * kBBuf;
        mbar_expect_tx(full, (uint32_t)bt.rows * kGatePairBytes);
        if (bt.rows == 64) bulk_copy(dst, src + bt.base, kBBuf, full);
        else                                              // the batch's last tile: shorter planes (what lies behind them is masked)
          for (int p = 0; p < 6; ++p) bulk_copy(dst + (uint32_t)p * 8192u, src + bt.base + (size_t)p * bt.rows * 128, (uint32_t)bt.rows * 128u, full);
        if (++buf == kBBufs) { buf = 0; ph ^= 1u; }
      }
    }
  } else if (warp >= 16) {
    // ------------------------------------------------------------------------------------------ MMAs
    // (the issuing threads copy nothing: a thread that waits for its own copies between two batches of MMAs leaves
    // the pipe idle for the latency of a copy, which was 40 % of the kernel)
    if (elect_one()) {
      const int part = warp - 16;                          // 0: small terms, 1: large terms
      // (A plane, B plane): small = (hi, lo), (lo, hi), (mid, mid); large = (hi, mid), (mid, hi), (hi, hi)
      const uint32_t pa[3] = {0u, part ? 1u : 2u, part ? 0u : 1u}, pb[3] = {part ? 1u : 2u, 0u, part ? 0u : 1u};
      uint32_t buf = 0, ph = 0, uses[2] = {0u, 0u};
      wait_bar(bar0 + 8 * A_FULL, 0u, abort_addr, status);
      for (int n = 0; n < products; ++n) {
        const int acc = (tile_lo + (n >= ntiles ? n - ntiles : n)) & 1;
        wait_bar(bar0 + 8 * (B_FULL + buf), ph, abort_addr, status);
        // the rows have taken the previous tile out of this accumulator pair
        const uint32_t use = acc ? uses[1]++ : uses[0]++;
        wait_bar(bar0 + 8 * (ACC_EMPTY + acc), (use & 1u) ^ 1u, abort_addr, status);
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)acc * 2u * kCols + (uint32_t)part * kCols;
        const uint32_t sb = base + buf * kBBuf;
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            tc_mma_ts(d, tmem + kColA + pa[t] * 64u + (uint32_t)kk * 8u,
                      make_desc(sb + pb[t] * kBPlane + (uint32_t)(kk >> 2) * (kCols * 128u) + (uint32_t)(kk & 3) * 32u, 16, 1024), kIdesc, (t | kk) != 0 ? 1u : 0u);
        tc_commit(bar0 + 8 * (B_EMPTY + buf));
        tc_commit(bar0 + 8 * (ACC_FULL + acc));
        if (++buf == kBBufs) { buf = 0; ph ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------------------------------ rows
    // everything in units of log2: x2 = logit * log2(e); m the running maximum of x2; p = 2^(x2 - m) / l
    const float scale2 = rsqrtf((float)kGateDim) * 1.4426950408889634f;
    float seg_m = -CUDART_INF_F, seg_l = 0.f;             // this thread's columns of the current segment
    float row_m = -CUDART_INF_F, row_l = 0.f, inv_l = 0.f;   // the whole row
    float2* ml = reinterpret_cast<float2*>(smem + kOffSeg);
    int nseg = 0;
    uint32_t uses = 0;                                    // tiles this group has worked on
    const uint32_t base4 = (uint32_t)(reinterpret_cast<uintptr_t>(scores) >> 2);   // scores may begin on any four bytes
    if (kMode == kWrite && my_last >= 0) {
      gate_row_stats(m, stats, h, my_last, my_start, row_m, row_l);
      inv_l = row_l > 0.f ? 1.0f / row_l : 0.f;
    }
    float x[32];
    for (int n = 0; n < total; ++n) {
      const bool write = kMode == kWrite || (kMode == kBoth && n >= ntiles);
      const int ct = tile_lo + (kMode == kBoth && n >= ntiles ? n - ntiles : n);
      const int j0 = ct * kCols + half * 32;              // first column of this thread
      if (kMode == kBoth && n == ntiles) inv_l = row_l > 0.f ? 1.0f / row_l : 0.f;
      if ((ct & 1) == grp) {
      if (!kept || n < ntiles) {
        wait_bar(bar0 + 8 * (ACC_FULL + grp), uses & 1u, abort_addr, status);
        ++uses;
        tc_fence_after();
        const uint32_t a = tmem + lane_addr + (uint32_t)grp * 2u * kCols + (uint32_t)half * 32u;
        uint32_t vs[32], vl[32];
        tc_ld32(a, vs);
        tc_ld32(a + kCols, vl);
        tc_wait_ld32(vs);
        tc_wait_ld32(vl);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar0 + 8 * (ACC_EMPTY + grp));
#pragma unroll
        for (int c = 0; c < 32; ++c) x[c] = __fmul_rn(__fadd_rn(__uint_as_float(vs[c]), __uint_as_float(vl[c])), scale2);
      }
      // columns that are causal for this row: j in [my_start, my_last]
      const int lo = my_start - j0, hi = my_last - j0;
      if (!write) {                                        // statistics
        if (hi >= 0 && lo <= 31) {
          if (lo > 0 || hi < 31) {
#pragma unroll
            for (int c = 0; c < 32; ++c) if (c < lo || c > hi) x[c] = -CUDART_INF_F;
          }
          float mx[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
          for (int c = 4; c < 32; ++c) mx[c & 3] = fmaxf(mx[c & 3], x[c]);
          const float nm = fmaxf(seg_m, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
          const float ref = fmaxf(nm, -CUDART_MAX_NORMAL_F);   // (nm = -inf: nothing but logits below the range of fp32 so far)
          float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int c = 0; c < 32; ++c) sum[c & 3] = __fadd_rn(sum[c & 3], ex2f(__fsub_rn(x[c], ref)));   // 2^(-inf) = 0 for the masked columns
          const float s4 = __fadd_rn(__fadd_rn(sum[0], sum[1]), __fadd_rn(sum[2], sum[3]));
          seg_l = __fadd_rn(__fmul_rn(seg_l, ex2f(__fsub_rn(seg_m, ref))), s4);              // 2^(-inf) = 0 on the first contribution
          seg_m = nm;
        }
      }
      if (write || kMode == kLogits) {
        if (write) {
#pragma unroll
          for (int c = 0; c < 32; ++c) x[c] = gate_score(x[c], row_m, inv_l);
        }
        float* stage = reinterpret_cast<float*>(smem + kOffStage) + warp * 1024;
#pragma unroll
        for (int c = 0; c < 32; c += 4)
          *reinterpret_cast<float4*>(stage + lane * 32 + (((c >> 2) ^ (lane & 7)) << 2)) = make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]);
        __syncwarp();
        // the warp's 32 rows, four rows per step: eight lanes take a row, a lane four consecutive columns of it
#pragma unroll 4
        for (int rr = 0; rr < 32; rr += 4) {
          const int lr = rr + (lane >> 3), mr = (warp & 3) * 32 + lr;
          const long long off = *reinterpret_cast<const long long*>(smem + kOffMeta + mr * 16);
          const int2 se = *reinterpret_cast<const int2*>(smem + kOffMeta + mr * 16 + 8);
          const int j = j0 + 4 * (lane & 7);
          const float4 v = *reinterpret_cast<const float4*>(stage + lr * 32 + (((lane & 7) ^ (lr & 7)) << 2));
          float* dst = scores + (off + j);
          if (j >= se.x && j + 3 <= se.y && (((uint32_t)off + base4) & 3u) == 0u) *reinterpret_cast<float4*>(dst) = v;   // (j is a multiple of four)
          else {
            if (j >= se.x && j <= se.y) dst[0] = v.x;
            if (j + 1 >= se.x && j + 1 <= se.y) dst[1] = v.y;
            if (j + 2 >= se.x && j + 2 <= se.y) dst[2] = v.z;
            if (j + 3 >= se.x && j + 3 <= se.y) dst[3] = v.w;
          }
        }
        __syncwarp();                                    // the staging rows are free again
      }
      }
      if (!write && (n == ntiles - 1 || ((ct + 1) * kCols) % seg_cols == 0)) {
        // end of a segment: the four threads of a row combine their columns
        float2* buf = ml + (nseg & 1) * 4 * kRows;
        buf[(grp * 2 + half) * kRows + row] = make_float2(seg_m, seg_l);
        named_bar_sync(1, kRowThreads);
        float sm = -CUDART_INF_F, sl = 0.f;
#pragma unroll
        for (int p = 0; p < 4; ++p) { const float2 v = buf[p * kRows + row]; gate_combine(sm, sl, v.x, v.y); }
        const int seg = ct * kCols / seg_cols, s_lo = my_start / seg_cols;
        const bool mine = my_last >= 0 && seg >= s_lo && seg <= my_last / seg_cols;
        if (kMode == kStats || kMode == kLogits) {
          if (mine && half == 0 && grp == 0) stats[((size_t)h * m.total_blocks + r0 + row) * stat_segs + (seg - s_lo)] = make_float2(sm, sl);
        } else if (mine) gate_combine(row_m, row_l, sm, sl);
        seg_m = -CUDART_INF_F; seg_l = 0.f;
        ++nseg;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// part_tiles == 0: one CTA per row tile and head
static dim3 score_grid(const SeqMeta& m, const ScoreBand& band, int part_tiles) {
  const unsigned x = (unsigned)((band.blk_hi - band.blk_lo + gs::kRows - 1) / gs::kRows) * (unsigned)band.heads;
  if (part_tiles && m.batch == 1) {
    unsigned n = 0;
    for (int t = 0; t < (int)(x / band.heads); ++t) n += (unsigned)gs::part_count(band, t, part_tiles);
    return dim3(n * (unsigned)band.heads, 1);
  }
  // a row tile that starts in one sequence and ends in another may touch a tile's worth of columns more than the longest one
  const int cols = part_tiles * gs::kCols;
  return dim3(x, part_tiles ? (unsigned)((m.max_nb + gs::kRows + cols - 1) / cols + 1) : 1u);
}

// Whether the whole problem takes two launches (statistics, then scores) rather than one.  In units of a tile (about 1 us): one
// launch lasts as long as its longest CTA (both sweeps of the longest row) or its share of all tiles; two launches even that
// out but pay a CTA's start (about three tiles) per segment, twice.
bool gate_split(const SeqMeta& m, int num_sms) {
  const int64_t tiles = m.score_tiles;
  const int64_t longest = (m.max_nb + gs::kCols - 1) / gs::kCols, share = tiles / num_sms;
  const int seg = gate_seg_tiles(m.max_nb);
  const int64_t starts = 1 + tiles / seg / num_sms;
  const int64_t one = 2 * (longest > share ? longest : share), two = 2 * ((seg > share ? seg : share) + 3 * starts) + 3;
  return two < one;
}

// Whether bands of logits, `bands` of them, take less time than the statistics of all rows and then bands of scores, in the same units.  A
// part of the logits is a whole segment at least, so a band of few rows lasts as long as that (16 tiles beyond 2048 blocks), where
// one of scores is split by four; and a band's selection takes about 1.5 longer to form the scores.  (Start of a CTA three; 200 000
// tokens, 16 heads in bands of 8 MB: 5.0 ms by 112 bands of logits, 3.3 by scores; 262 144 tokens, 32 heads in 128 MB: 2.1 and 2.4.)
bool gate_logits_pay(const SeqMeta& m, int64_t bands, int num_sms) {
  const double tiles = (double)m.score_tiles, sms = num_sms, seg = gate_seg_tiles(m.max_nb), longest = (m.max_nb + gs::kCols - 1) / gs::kCols;
  const auto launch = [&](double all, double part) { return std::max(all * (1.0 + 3.0 / part) / sms, std::min(part, longest) + 3.0); };
  double of_logits = 1e30, of_scores = 1e30;
  for (double p = seg; p < 2.0 * std::max(longest, seg); p *= 2.0) of_logits = std::min(of_logits, launch(tiles / (double)bands, p));
  for (double p = 4.0; p <= 16.0; p *= 2.0) of_scores = std::min(of_scores, launch(tiles / (double)bands, p));
  return (double)bands * (of_logits + 1.5 - of_scores) <= launch(tiles, seg) + 3.0;
}

// Statistics of all rows.
int launch_gate_stats(const SeqMeta& m, const uint16_t* gq, const uint16_t* gk, float2* stats, int* status, cudaStream_t stream) {
  const ScoreBand all = {m.first_q_block, m.total_blocks, 0, m.num_q_heads, 0, 0, 0};
  const int part = gate_seg_tiles(m.max_nb);
  const dim3 grid = score_grid(m, all, part);
  if (grid.x == 0) return 0;
  const cudaError_t e = launch_next(gate_scores_kernel<gs::kStats>, grid, gs::kThreads, gs::kSmemBytes, stream, m, all, gq, gk, nullptr, stats, status, part);
  return e == cudaSuccess ? 1 : -(int)e;
}

// Scores of a band; with `stats` launch_gate_stats has run, without the rows' statistics are formed by the same launch.
int launch_gate_scores(const SeqMeta& m, const ScoreBand& band, const uint16_t* gq, const uint16_t* gk, float* scores,
                       float2* stats, int* status, int num_sms, cudaStream_t stream) {
  // Parts of 4, 8 or 16 tiles: what lasts shortest, in units of a tile.  A CTA's start is about three of them; a launch lasts as long as
  // a full part or its share of all tiles and starts.  (128 rows of 32 heads against 2048 blocks: 8 tiles to a part instead of
  // 4: gate and mask of the chunk 170 -> 162 us; three 4096-block heads: 16, where 8 take 7 % longer.)
  int part = 4;
  if (stats != nullptr) {
    const dim3 all = score_grid(m, band, 1);
    const int64_t tiles = (int64_t)all.x * all.y;
    int64_t best = INT64_MAX;
    for (int p = 4; p <= 16; p *= 2) {
      const dim3 g = score_grid(m, band, p);
      const int64_t share = (tiles + 3 * (int64_t)g.x * g.y) / num_sms, cost = share > p + 3 ? share : p + 3;
      if (cost < best) { best = cost; part = p; }
    }
  }
  const dim3 grid = score_grid(m, band, stats != nullptr ? part : 0);
  if (grid.x == 0) return 0;
  const cudaError_t e = stats != nullptr
      ? launch_next(gate_scores_kernel<gs::kWrite>, grid, gs::kThreads, gs::kSmemBytes, stream, m, band, gq, gk, scores, stats, status, part)
      : launch_next(gate_scores_kernel<gs::kBoth>, grid, gs::kThreads, gs::kSmemBytes, stream, m, band, gq, gk, scores, nullptr, status, 0);
  return e == cudaSuccess ? 1 : -(int)e;
}

// Logits of a band and the statistics of its rows by one launch, for selection kernels that form the scores themselves.  Parts of 1, 2, 4 ..
// segments, or whole rows: what lasts shortest, by the same estimate.
int launch_gate_logits(const SeqMeta& m, const ScoreBand& band, const uint16_t* gq, const uint16_t* gk, float* logits, float2* stats,
                       int* status, int num_sms, cudaStream_t stream) {
  const dim3 all = score_grid(m, band, 1), rows = score_grid(m, band, 0);
  if (rows.x == 0) return 0;
  const int64_t tiles = (int64_t)all.x * all.y, longest = (m.max_nb + gs::kCols - 1) / gs::kCols;
  int part = 0;
  int64_t best = std::max((tiles + 3 * (int64_t)rows.x) / num_sms, longest + 3);
  for (int p = gate_seg_tiles(m.max_nb); p < longest; p *= 2) {
    const dim3 g = score_grid(m, band, p);
    const int64_t cost = std::max((tiles + 3 * (int64_t)g.x * g.y) / num_sms, (int64_t)p + 3);
    if (cost < best) { best = cost; part = p; }
  }
  const cudaError_t e = launch_next(gate_scores_kernel<gs::kLogits>, score_grid(m, band, part), gs::kThreads, gs::kSmemBytes, stream, m, band, gq, gk, logits, stats, status, part);
  return e == cudaSuccess ? 1 : -(int)e;
}

// Lifts the kernels' shared-memory limit on the current device (no allocation).
bool init_gate_scores() {
  return cudaFuncSetAttribute(gate_scores_kernel<gs::kBoth>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gs::kSmemBytes) == cudaSuccess &&
         cudaFuncSetAttribute(gate_scores_kernel<gs::kStats>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gs::kSmemBytes) == cudaSuccess &&
         cudaFuncSetAttribute(gate_scores_kernel<gs::kWrite>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gs::kSmemBytes) == cudaSuccess &&
         cudaFuncSetAttribute(gate_scores_kernel<gs::kLogits>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gs::kSmemBytes) == cudaSuccess;
}

}  // namespace seer
