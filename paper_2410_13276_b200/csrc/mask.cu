// Binary block mask (Sec. 3.3, Eq. 3 TopK / Eq. 4 threshold) as CSR index lists.
//   count_kernel : one warp per (sequence, head, query-block) row -> number of kept blocks
//   scan_kernel  : exclusive prefix sum of the counts -> row_ptr, nnz, capacity check
//   topk_kernel / fill_kernel : repeat the selection and write the ascending lists
// Selection order in the TopK modes is (score descending, block index ascending): scores become order-preserving
// 32-bit keys, the key of the last kept candidate is found (by bins of the keys' distance from the smallest in topk_kernel, by a radix
// select of at most four 8-bit passes in fill_kernel), and ties at that key are resolved by rank in index order.
#include <math_constants.h>

#include "seer_internal.cuh"

namespace seer {

constexpr int kMaskWarps = 4;
// TopK rows of up to this many blocks are held in shared memory (topk_kernel); longer ones re-read their scores in every pass.
constexpr int kTopkRowMax = 16384;

struct RowInfo {
  const float* s;   // scores of this row
  int i;            // query block index (row has n = i + 1 causal blocks)
  bool valid;
  bool skip;        // chunked prefill: a query block before the chunk, its list is empty
  int nb;           // blocks of the row's sequence
  int h, gb;        // head; block row, numbered over the batch
};

// Rows [row_lo, row_hi) of the CSR structure and where their scores are (ScoreBand).
struct RowBand {
  int64_t row_lo, row_hi;
  ScoreBand sb;
};

__device__ __forceinline__ RowInfo decode_row(const SeqMeta& m, const RowBand& band, const float* scores, int64_t r) {
  RowInfo ri;
  ri.valid = r < band.row_hi;
  ri.skip = false;
  ri.nb = 0;
  if (!ri.valid) { ri.s = nullptr; ri.i = 0; return ri; }
  // (the host refuses shapes with 2^31 rows or more: 32-bit divisions)
  const int b = find_sequence(m.blk_off, m.batch, (int)((uint32_t)r / (uint32_t)m.num_q_heads));
  const int nb = m.blk_off[b + 1] - m.blk_off[b];
  const uint32_t local = (uint32_t)r - (uint32_t)m.num_q_heads * (uint32_t)m.blk_off[b];
  const int h = (int)(local / (uint32_t)nb);
  ri.i = (int)(local - (uint32_t)h * (uint32_t)nb);
  ri.s = scores + score_row_offset(m, band.sb, b, nb, h, ri.i);   // (not looked at for a skipped row)
  ri.skip = m.chunked && ri.i < m.qoff[b];
  ri.nb = nb;
  ri.h = h;
  ri.gb = m.blk_off[b] + ri.i;
  return ri;
}

// Order-preserving map fp32 -> uint32 (larger score = larger key); -0 equals +0; NaN -> 0 (never a candidate).
__device__ __forceinline__ uint32_t score_key(float s) {
  uint32_t u = __float_as_uint(s);
  if ((u & 0x7fffffffu) > 0x7f800000u) return 0u;
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ bool is_forced(int j, int i, uint32_t flags) {
  return ((flags & SEER_FORCE_DIAG) && j == i) || ((flags & SEER_FORCE_SINK) && j == 0);
}

__device__ __forceinline__ int num_forced(int i, uint32_t flags) {
  int nf = (flags & SEER_FORCE_DIAG) ? 1 : 0;
  if ((flags & SEER_FORCE_SINK) && !((flags & SEER_FORCE_DIAG) && i == 0)) nf += 1;
  return nf;
}

__device__ __forceinline__ int keep_count(int n, const seer_mask_params& p) {
  if (p.mode == SEER_TOPK_RATIO) {
    long long k = ((long long)p.keep_num * n + p.keep_den - 1) / p.keep_den;
    if (k < 1) k = 1;
    if (k > n) k = n;
    return (int)k;
  }
  int k = p.k < 0 ? 0 : p.k;
  return k < n ? k : n;
}

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(kMaskWarps * 32)
count_kernel(SeqMeta m, RowBand band, const float* scores, seer_mask_params p, int32_t* row_ptr) {
  const int lane = threadIdx.x & 31;
  const int64_t r = band.row_lo + (int64_t)blockIdx.x * kMaskWarps + (threadIdx.x >> 5);
  const RowInfo ri = decode_row(m, band, scores, r);
  grid_wait();
  if (!ri.valid) return;
  const int n = ri.i + 1;
  int c = 0;
  if (ri.skip) {
    // nothing listed
  } else if (ri.i >= ri.nb - p.dense_tail_blocks) {
    c = n;                                             // a dense row at the end of the sequence
  } else if (p.mode == SEER_THRESHOLD) {
    int head = 0;
    if ((reinterpret_cast<uintptr_t>(ri.s) & 15) == 0) {       // four scores per lane and load where the row is aligned
      head = n & ~3;
      for (int j = lane * 4; j < head; j += 128) {
        const float4 v = *reinterpret_cast<const float4*>(ri.s + j);
        c += (is_forced(j, ri.i, p.flags) || v.x > p.threshold) ? 1 : 0;
        c += (is_forced(j + 1, ri.i, p.flags) || v.y > p.threshold) ? 1 : 0;
        c += (is_forced(j + 2, ri.i, p.flags) || v.z > p.threshold) ? 1 : 0;
        c += (is_forced(j + 3, ri.i, p.flags) || v.w > p.threshold) ? 1 : 0;
      }
    }
    for (int j = head + lane; j < n; j += 32) c += (is_forced(j, ri.i, p.flags) || ri.s[j] > p.threshold) ? 1 : 0;
    c = warp_sum(c);
  } else {
    int head = 0;
    if ((reinterpret_cast<uintptr_t>(ri.s) & 15) == 0) {
      head = n & ~3;
      for (int j = lane * 4; j < head; j += 128) {
        const float4 v = *reinterpret_cast<const float4*>(ri.s + j);
        c += (!is_forced(j, ri.i, p.flags) && score_key(v.x) != 0u) ? 1 : 0;
        c += (!is_forced(j + 1, ri.i, p.flags) && score_key(v.y) != 0u) ? 1 : 0;
        c += (!is_forced(j + 2, ri.i, p.flags) && score_key(v.z) != 0u) ? 1 : 0;
        c += (!is_forced(j + 3, ri.i, p.flags) && score_key(v.w) != 0u) ? 1 : 0;
      }
    }
    for (int j = head + lane; j < n; j += 32) c += (!is_forced(j, ri.i, p.flags) && score_key(ri.s[j]) != 0u) ? 1 : 0;
    const int ncand = warp_sum(c);
    const int nf = num_forced(ri.i, p.flags);
    const int take = max(keep_count(n, p) - nf, 0);
    c = nf + min(take, ncand);
  }
  if (lane == 0) row_ptr[r + 1] = c;
}

// TopK counts of scores whose softmax statistics are at hand, four threads a row.  A row whose maximum and sum are finite has no
// NaN among its scores, so its length follows from n and the parameters and no score is read (4096 rows of 4096 blocks: 15 us
// with count_kernel); a row that has not is counted by its threads (kLogits: from the scores that the selection will form).  Gate + mask of
// rows that are all spoilt, by one thread each and so: 32k tokens, 32 heads 183 and 136 us, 128k 5.65 and 1.11 ms
// (a warp a row after the other: 145 us and 0.91 ms, but 8k tokens 62 where this takes 52).
template <bool kLogits>
__global__ void __launch_bounds__(128)
topk_count_kernel(SeqMeta m, RowBand band, const float* scores, const float2* stats, seer_mask_params p,
                  int32_t* row_ptr) {
  const int sub = threadIdx.x & 3;
  const int64_t r = band.row_lo + (int64_t)blockIdx.x * 32 + (threadIdx.x >> 2);
  const RowInfo ri = decode_row(m, band, scores, r);
  grid_wait();
  const int n = ri.i + 1;
  int nf = 0, take = 0, c = 0;
  bool spoilt = false;
  float row_m = 0.f, inv_l = 0.f;
  if (!ri.valid || ri.skip) {
    // nothing listed
  } else if (ri.i >= ri.nb - p.dense_tail_blocks) {
    c = n;
  } else {
    nf = num_forced(ri.i, p.flags);
    take = max(keep_count(n, p) - nf, 0);
    const int seg_cols = gate_seg_tiles(m.max_nb) * kScoreTile, segs = ri.gb / seg_cols - (ri.gb - ri.i) / seg_cols + 1;
    const float2* st = stats + ((size_t)ri.h * m.total_blocks + ri.gb) * gate_stat_segs(m.max_nb);
    for (int s = 0; s < segs; ++s) { const float2 v = st[s]; spoilt = spoilt || !(fabsf(v.x) < 3.0e38f && v.y > 0.f && v.y < 3.0e38f); }
    c = nf + min(take, n - nf);
  }
  if (__any_sync(0xffffffffu, spoilt)) {
    int ncand = 0;
    if (spoilt) {
      if (kLogits) {
        float row_l = 0.f;
        gate_row_stats(m, stats, ri.h, ri.gb, ri.gb - ri.i, row_m, row_l);
        inv_l = row_l > 0.f ? 1.0f / row_l : 0.f;
      }
#pragma unroll 8
      for (int j = sub; j < n; j += 4) {
        const float x = kLogits ? gate_score(ri.s[j], row_m, inv_l) : ri.s[j];
        ncand += (!is_forced(j, ri.i, p.flags) && score_key(x) != 0u) ? 1 : 0;
      }
    }
    ncand += __shfl_xor_sync(0xffffffffu, ncand, 1);
    ncand += __shfl_xor_sync(0xffffffffu, ncand, 2);
    if (spoilt) c = nf + min(take, ncand);
  }
  if (ri.valid && sub == 0) row_ptr[r + 1] = c;
}

// In-place inclusive scan of row_ptr[1..rows] by one CTA or a cluster of eight.  `first`: row_ptr[0] = 0; otherwise the scan
// continues from row_ptr[0], the last entry of the rows scanned before.  Tiles of 8192 counts go through shared memory (coalesced
// loads and stores, the next tile's loads in flight meanwhile), eight consecutive counts per thread, warp shuffles inside a
// warp; every warp adds up the warp totals for itself, every CTA the tile totals that the others have put into its shared memory.
// A CTA alone is bound by the latency of a tile's three barriers, about 2 us a tile; beyond one tile the cluster takes eight at a time
// (counts, scan and lists of 76 800 rows: 123 us by one CTA, 111 so).  All sums fit 32 bits, unsigned: the host
// refuses shapes with 2^31 causal blocks, and lists to be expanded may hold entries past the diagonal, twice as many at most.
constexpr int kScanPer = 8, kScanTile = 1024 * kScanPer, kScanRanks = 8;
template <int kRanks>
__global__ void __launch_bounds__(1024)
scan_kernel(int64_t rows, int32_t* row_ptr, int first, int64_t col_capacity, int64_t* __restrict__ nnz_out,
            int* __restrict__ status) {
  __shared__ int32_t tile[kScanTile + kScanTile / 32];     // (one word of padding per 32: eight consecutive words per thread)
  __shared__ uint32_t warp_tot[2][32], rank_tot[2][kRanks];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rank = kRanks > 1 ? (int)blockIdx.x : 0;       // (the grid is one cluster)
  grid_wait();
  uint32_t carry = first ? 0u : (uint32_t)__ldcg(row_ptr); // (read past L1: the kernel rewrites it)
  int32_t next[kScanPer];
#pragma unroll
  for (int k = 0; k < kScanPer; ++k) {
    const int64_t idx = (int64_t)rank * kScanTile + t + k * 1024;
    next[k] = idx < rows ? __ldcg(row_ptr + idx + 1) : 0;
  }
  // (a CTA's shared memory may be written to once it runs)
  if (kRanks > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  int par = 0;
  for (int64_t base0 = 0; base0 < rows; base0 += kRanks * kScanTile, par ^= 1) {
    const int64_t base = base0 + rank * kScanTile;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) { const int idx = t + k * 1024; tile[idx + (idx >> 5)] = next[k]; }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int64_t idx = base + kRanks * kScanTile + t + k * 1024;
      next[k] = idx < rows ? __ldcg(row_ptr + idx + 1) : 0;
    }
    uint32_t v[kScanPer];
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) { const int idx = kScanPer * t + k; v[k] = (uint32_t)tile[idx + (idx >> 5)] + (k > 0 ? v[k - 1] : 0u); }
    uint32_t incl = v[kScanPer - 1];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) warp_tot[par][warp] = incl;
    __syncthreads();
    uint32_t w = warp_tot[par][lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += o;
    }
    const uint32_t before_warp = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
    uint32_t total = __shfl_sync(0xffffffffu, w, 31);
    if (kRanks > 1) {
      if (t < kRanks) {                                    // this CTA's total to CTA t
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&rank_tot[par][rank]);
        uint32_t theirs;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(t));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(theirs), "r"(total) : "memory");
      }
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      total = 0;
#pragma unroll
      for (int q = 0; q < kRanks; ++q) {
        const uint32_t x = rank_tot[par][q];
        if (q < rank) carry += x; else total += x;         // (carry: counts before this CTA's tile)
      }
    }
    const uint32_t before = carry + (warp > 0 ? before_warp : 0u) + (incl - v[kScanPer - 1]);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) { const int idx = kScanPer * t + k; tile[idx + (idx >> 5)] = (int32_t)(before + v[k]); }
    carry += total;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int idx = t + k * 1024;
      if (base + idx < rows) row_ptr[base + idx + 1] = tile[idx + (idx >> 5)];
    }
    // (a thread's stores of the next tile go to the words it has just read)
  }
  if (t == 0 && rank == 0) {
    if (first) row_ptr[0] = 0;
    if (nnz_out) *nnz_out = (int64_t)carry;
    if ((int64_t)carry > col_capacity) atomicCAS(status, 0, (int)SEER_ERR_CAPACITY);
  }
}

// Counts and their scan by one CTA, for masks of few short rows: the two kernels are a launch and a few latencies each, and there is nothing
// else to do meanwhile.  Eight lanes take a row, 128 rows go at a time, and each pass begins with the rows' addresses: past two to four of
// them the one CTA is the slower way.  Mask alone, two kernels and this, one to sixteen sequences: 256 rows of 64 blocks, TopK 9.9 and
// 8.1 to 8.5 us; 384 of 48 9.9 and 9.2 to 9.9; 384 of 64 10.0 and 10.0 to 10.6; 512 of 32 10.1 and 11.3 to 11.9.  Thresholds take fewer instructions
// an entry: 384 of 64 9.8 and 8.6 to 9.1, 512 of 32 10.1 and 8.9 to 9.7, 512 of 64 9.7 and 10.3 to 11.4.
constexpr int kSmallRows = 512, kSmallBlocks = 64;
static bool small_mask(int64_t rows, int max_nb, int mode) {
  if (max_nb > kSmallBlocks) return false;
  return rows <= (mode == SEER_THRESHOLD ? (max_nb <= 32 ? kSmallRows : 384) : max_nb <= 48 ? 384 : 256);
}
__global__ void __launch_bounds__(1024)
count_scan_kernel(SeqMeta m, RowBand band, const float* scores, seer_mask_params p, int32_t* row_ptr, int first, int64_t col_capacity,
                  int64_t* __restrict__ nnz_out, int* __restrict__ status) {
  __shared__ uint32_t counts[kSmallRows], warp_tot[kSmallRows / 32];
  const int t = threadIdx.x, lane = t & 31, sub = t & 7, rows = (int)(band.row_hi - band.row_lo);
  RowInfo ri = decode_row(m, band, scores, band.row_lo + (t >> 3));
  grid_wait();
  const uint32_t carry = first ? 0u : (uint32_t)__ldcg(row_ptr + band.row_lo);   // (read past L1: the kernel before may have written it)
  for (int r0 = 0; r0 < rows; r0 += 128) {
    if (r0 > 0) ri = decode_row(m, band, scores, band.row_lo + r0 + (t >> 3));
    const int n = ri.i + 1;
    const bool dense = ri.i >= ri.nb - p.dense_tail_blocks, looked_at = ri.valid && !ri.skip && !dense;
    int c = 0;
    if (looked_at) {
#pragma unroll 8
      for (int j = sub; j < n; j += 8) {
        const float x = ri.s[j];
        const bool forced = is_forced(j, ri.i, p.flags);
        c += p.mode == SEER_THRESHOLD ? forced || x > p.threshold : !forced && score_key(x) != 0u;
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (looked_at && p.mode != SEER_THRESHOLD) {
      const int nf = num_forced(ri.i, p.flags);
      c = nf + min(max(keep_count(n, p) - nf, 0), c);
    }
    if (ri.valid && sub == 0) counts[r0 + (t >> 3)] = (uint32_t)(ri.skip ? 0 : dense ? n : c);
  }
  __syncthreads();
  uint32_t incl = t < rows ? counts[t] : 0u;
  if (t < kSmallRows) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) warp_tot[t >> 5] = incl;
  }
  __syncthreads();
  if (t >= rows) return;
  uint32_t before = carry;
  for (int w = 0; w < t >> 5; ++w) before += warp_tot[w];
  row_ptr[band.row_lo + t + 1] = (int32_t)(before + incl);
  if (t == 0 && first) row_ptr[band.row_lo] = 0;
  if (t == rows - 1) {
    if (nnz_out) *nnz_out = (int64_t)(before + incl);
    if ((int64_t)(before + incl) > col_capacity) atomicCAS(status, 0, (int)SEER_ERR_CAPACITY);
  }
}

static cudaError_t launch_scan(int64_t rows, int32_t* row_ptr, int first, int64_t col_capacity, int64_t* nnz_out, int* status,
                               cudaStream_t stream) {
  if (rows <= kScanTile)
    return launch_next(scan_kernel<1>, 1, 1024, 0, stream, rows, row_ptr, first, col_capacity, nnz_out, status);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kScanRanks);
  cfg.blockDim = dim3(1024);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kScanRanks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, scan_kernel<kScanRanks>, rows, row_ptr, first, col_capacity, nnz_out, status);
}

// The key a TopK row is ranked by, in fewer instructions than score_key (the loops are bound by instruction issue).
__device__ __forceinline__ uint32_t lean_key(float sc) {
  const float z = sc + 0.0f;                                     // -0 -> +0
  const uint32_t u = __float_as_uint(z);
  const uint32_t kk = u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
  return z != z ? 0u : kk;                                       // NaN: never a candidate
}

// TopK lists, W = 1, 4 or 8 warps per row, the row's keys in shared memory (`cap` of them, a multiple of 128 W).  A warp works on a contiguous
// run of the row's columns, 128 at a time, a lane four of them.
//
// It is bound by instruction issue (three of four per clock on average, four warps a row), so the loops are short and rolled (with the keys in registers and the
// loops unrolled it waited for instructions), what a row needs once is done by one of its warps and passed on, and the
// counts that order the warps' parts of the list are taken in the pass that gathers the threshold's class.
// A row gets one warp up to 2048 blocks, and as many as keep it at 2048 keys per warp beyond.  Measured: 65 536 rows of up to
// 2048 blocks 176 us, 4096 rows of up to 4096 blocks 31 us (fill_kernel, which re-reads the scores in every pass: 158); what a row
// needs once done by every warp of it, and a pass of its own for the counts: 183 and 34.
//
// kLogits: the rows hold logits in units of log2, not scores; `stats` are the softmax statistics of the row's segments.  A score
// is formed here as the score kernel forms it, bit for bit.
template <int W, bool kLogits>
__global__ void __launch_bounds__(W == 1 ? 128 : W * 32, W < 8 ? 12 : 6)
topk_kernel(SeqMeta m, RowBand band, const float* scores, const float2* stats, seer_mask_params p, const int32_t* row_ptr,
            int32_t* col_idx, int64_t col_capacity, int cap) {
  static_assert(W == 1 || W == 4 || W == 8, "a row has a warp or a CTA to itself");
  constexpr int kRows = W == 1 ? 4 : 1;
  extern __shared__ __align__(16) uint32_t key_smem[];
  __shared__ __align__(16) uint32_t s_hist[kRows][256];
  __shared__ uint32_t s_red[kRows][3][W];
  __shared__ uint32_t s_list[kRows][32];
  __shared__ uint32_t s_own[kRows][32];
  __shared__ uint32_t s_found[kRows];
  __shared__ int s_cnt[kRows][2][W];
  __shared__ uint32_t s_pick[kRows][4];
  __shared__ RowInfo s_row[kRows];
  __shared__ float s_stat[kRows][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rr = warp / W, w = warp % W;                         // row of the CTA, warp within the row's group
  auto meet = [&]() {                                            // the warps of a row
    if (W == 1) __syncwarp();
    else __syncthreads();
  };
  const int64_t r = band.row_lo + (int64_t)blockIdx.x * kRows + rr;
  RowInfo ri;
  if (W == 1 || w == 0) {
    ri = decode_row(m, band, scores, r);
    if (W > 1 && lane == 0) s_row[rr] = ri;
  }
  grid_wait();
  float row_m = 0.f, row_l = 0.f;
  if (kLogits && (W == 1 || w == 0) && ri.valid && !ri.skip) {
    gate_row_stats(m, stats, ri.h, ri.gb, ri.gb - ri.i, row_m, row_l);
    if (W > 1 && lane == 0) { s_stat[rr][0] = row_m; s_stat[rr][1] = row_l; }
  }
  if (W > 1) {
    meet();
    ri = s_row[rr];
    if (kLogits) { row_m = s_stat[rr][0]; row_l = s_stat[rr][1]; }
  }
  if (!ri.valid || ri.skip) return;                              // (uniform in a row's group)
  const int n = ri.i + 1;
  const int32_t out0 = row_ptr[r], out1 = row_ptr[r + 1];
  if ((int64_t)out1 > col_capacity) return;   // this row (and all later ones) do not fit; status already raised
  int32_t* out = col_idx + out0;
  const uint32_t lt_mask = (1u << lane) - 1u;
  if (ri.i >= ri.nb - p.dense_tail_blocks) {           // a dense row at the end of the sequence: every causal block
    for (int j = w * 32 + lane; j < n; j += W * 32) out[j] = j;
    return;
  }
  uint32_t* keys = key_smem + (size_t)rr * cap;
  uint32_t* hist = s_hist[rr];
  const bool sink_f = (p.flags & SEER_FORCE_SINK) != 0u;
  const bool diag_f = (p.flags & SEER_FORCE_DIAG) != 0u && !(sink_f && ri.i == 0);
  const int take = max(keep_count(n, p) - num_forced(ri.i, p.flags), 0);
  const int run_cols = (n + 128 * W - 1) / (128 * W) * 128;      // columns of a warp
  const int j_lo = w * run_cols, j_hi = min(j_lo + run_cols, n), j_mine = j_lo + 4 * lane;

  // ---- keys (0: not a candidate: past the row, NaN, or forced, which the writer puts in its place by itself)
  uint32_t c = 0, k_min = 0xffffffffu, k_max = 0u;               // over the candidates
  const uint32_t nan_bits = 0x7fffffffu;
  const float inv_l = row_l > 0.f ? 1.0f / row_l : 0.f;
  auto key_of = [&](uint32_t raw) -> uint32_t { return lean_key(kLogits ? gate_score(__uint_as_float(raw), row_m, inv_l) : __uint_as_float(raw)); };
  const uint32_t* src = reinterpret_cast<const uint32_t*>(ri.s);
  const bool vec = (reinterpret_cast<uintptr_t>(ri.s) & 15) == 0;
  // A row whose statistics are finite has no NaN among its scores, and none below zero: every column but the forced ones is a candidate, and a
  // score's bits rank it.  (Gate and lists of 262 144 tokens, 32 heads, one in twenty 2107 us without this and with the statistics read by every warp
  // of a row, 2020 so.  A warp by itself has no registers for the second form of the loop: 131 072 tokens 671 and 673.)
  const bool clean = kLogits && W > 1 && fabsf(row_m) < 3.0e38f && row_l > 0.f && row_l < 3.0e38f;
  const int j_end = diag_f ? min(j_hi, ri.i) : j_hi;             // (the diagonal is a row's last column)
  if (clean && w == 0 && lane == 0) c = (uint32_t)(n - num_forced(ri.i, p.flags));
  auto plain_key = [&](uint32_t raw) -> uint32_t { return __float_as_uint(gate_score(__uint_as_float(raw), row_m, inv_l)) | 0x80000000u; };
  for (int j0 = j_mine; j0 - 4 * lane < j_hi; j0 += 512) {
    uint4 v[4];                                                  // four loads in flight per lane
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + q * 128;
      v[q] = make_uint4(nan_bits, nan_bits, nan_bits, nan_bits);
      if (vec && j + 3 < j_hi) v[q] = ld_global_v4(src + j);
      else if (j < j_hi) {
        v[q].x = ld_global(src + j);
        if (j + 1 < j_hi) v[q].y = ld_global(src + j + 1);
        if (j + 2 < j_hi) v[q].z = ld_global(src + j + 2);
        if (j + 3 < j_hi) v[q].w = ld_global(src + j + 3);
      }
    }
    if (clean) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = j0 + q * 128;
        if (j - 4 * lane >= j_hi) break;                         // (uniform)
        uint4 kq = make_uint4(plain_key(v[q].x), plain_key(v[q].y), plain_key(v[q].z), plain_key(v[q].w));
        if ((sink_f && j == 0) || j + 3 >= j_end) {              // not all four are candidates
          if (j >= j_end || (sink_f && j == 0)) kq.x = 0u;
          if (j + 1 >= j_end) kq.y = 0u;
          if (j + 2 >= j_end) kq.z = 0u;
          if (j + 3 >= j_end) kq.w = 0u;
          k_min = min(min(k_min, min(kq.x - 1u, kq.y - 1u)), min(kq.z - 1u, kq.w - 1u));   // (0 wraps to the largest)
        } else k_min = min(k_min, min(min(kq.x, kq.y), min(kq.z, kq.w)) - 1u);
        *reinterpret_cast<uint4*>(keys + j) = kq;
        k_max = max(max(k_max, max(kq.x, kq.y)), max(kq.z, kq.w));
      }
      continue;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + q * 128;
      if (j - 4 * lane >= j_hi) break;                           // (uniform)
      uint4 kq = make_uint4(key_of(v[q].x), key_of(v[q].y), key_of(v[q].z), key_of(v[q].w));
      if (sink_f && j == 0) kq.x = 0u;
      if (diag_f && (uint32_t)(ri.i - j) < 4u) {
        if (j == ri.i) kq.x = 0u;
        if (j + 1 == ri.i) kq.y = 0u;
        if (j + 2 == ri.i) kq.z = 0u;
        if (j + 3 == ri.i) kq.w = 0u;
      }
      *reinterpret_cast<uint4*>(keys + j) = kq;
      c += (kq.x != 0u) + (kq.y != 0u) + (kq.z != 0u) + (kq.w != 0u);
      k_max = max(max(k_max, max(kq.x, kq.y)), max(kq.z, kq.w));
      k_min = min(min(k_min, min(kq.x - 1u, kq.y - 1u)), min(kq.z - 1u, kq.w - 1u));   // (0, not a candidate, wraps to the largest)
    }
  }
  auto clear_hist = [&]() {
    *reinterpret_cast<uint4*>(hist + lane * 8) = make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(hist + lane * 8 + 4) = make_uint4(0u, 0u, 0u, 0u);
  };
  if (w == 0) {
    clear_hist();
    if (lane == 0) s_found[rr] = 0u;
  }
  uint32_t ncand = __reduce_add_sync(0xffffffffu, c);
  k_min = __reduce_min_sync(0xffffffffu, k_min);
  k_max = __reduce_max_sync(0xffffffffu, k_max);
  if (W > 1) {
    if (lane == 0) { s_red[rr][0][w] = ncand; s_red[rr][1][w] = k_min; s_red[rr][2][w] = k_max; }
    meet();
    ncand = __reduce_add_sync(0xffffffffu, lane < W ? s_red[rr][0][lane % W] : 0u);
    k_min = __reduce_min_sync(0xffffffffu, lane < W ? s_red[rr][1][lane % W] : 0xffffffffu);
    k_max = __reduce_max_sync(0xffffffffu, lane < W ? s_red[rr][2][lane % W] : 0u);
  } else meet();

  // ---- T: kept are the candidates with key >= T, of those with key == T only the first need_eq of n_eq
  uint32_t T = 1u;
  int need_eq = 0, n_eq = 0;
  bool counted = W == 1;                                         // s_cnt[.][0] holds the warps' kept columns
  if (take >= (int)ncand) {
    // every candidate is kept
  } else if (take == 0) {
    T = 0xffffffffu;                // nothing beyond the forced blocks (no key is that large: it would be a NaN's)
  } else {
    // The scores of a row are close together (probabilities of one softmax), often on both sides of a power of two.  So the
    // first pass bins the distance from the smallest key, scaled to 128..256 bins: binning the keys' own leading bits put a
    // flat row into a dozen bins, 32 lanes adding to a few shared-memory words, and took another pass.
    uint32_t lo = k_min + 1u, span = k_max - lo;                          // the class: keys lo .. lo + span
    int shift = max(24 - __clz(span | 1u), 0);
    int remaining = take;           // rank (1-based, from the top) still to locate inside the current class
    for (;;) {
      for (int j = j_mine; j - 4 * lane < j_hi; j += 128) {
        const uint4 kq = *reinterpret_cast<const uint4*>(keys + j);
        if (kq.x - lo <= span) atomicAdd(&hist[(kq.x - lo) >> shift], 1u);
        if (kq.y - lo <= span) atomicAdd(&hist[(kq.y - lo) >> shift], 1u);
        if (kq.z - lo <= span) atomicAdd(&hist[(kq.z - lo) >> shift], 1u);
        if (kq.w - lo <= span) atomicAdd(&hist[(kq.w - lo) >> shift], 1u);
      }
      meet();
      uint32_t found = 0u;                               // digit that holds the rank sought, its keys and the rank within them
      int cls = 0;
      if (W == 1 || w == 0) {
        // lane l owns digits 8l .. 8l+7; suffix sums over lanes give the number of keys with a larger digit
        uint32_t b[8], lane_total = 0u;
        {
          const uint4 h0 = *reinterpret_cast<const uint4*>(hist + lane * 8), h1 = *reinterpret_cast<const uint4*>(hist + lane * 8 + 4);
          b[0] = h0.x; b[1] = h0.y; b[2] = h0.z; b[3] = h0.w; b[4] = h1.x; b[5] = h1.y; b[6] = h1.z; b[7] = h1.w;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) lane_total += b[e];
        uint32_t above = lane_total;                     // inclusive suffix sum over lanes >= this lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t x = __shfl_down_sync(0xffffffffu, above, o);
          if (lane + o < 32) above += x;
        }
        above -= lane_total;                             // keys in lanes with larger digits
        // the digit holding rank `remaining` lies in the lane where above < remaining <= above + lane_total
        const bool mine = (int)above < remaining && remaining <= (int)(above + lane_total);
        int rank = 0;
        if (mine) {
          uint32_t acc = above;
#pragma unroll
          for (int e = 7; e >= 0; --e) {
            if ((int)acc < remaining && remaining <= (int)(acc + b[e])) { found = (uint32_t)(lane * 8 + e); rank = remaining - (int)acc; cls = (int)b[e]; }
            acc += b[e];
          }
        }
        if (W > 1) {
          clear_hist();
          if (mine) { s_pick[rr][0] = found; s_pick[rr][1] = (uint32_t)rank; s_pick[rr][2] = (uint32_t)cls; }
        } else {
          const int at = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
          found = __shfl_sync(0xffffffffu, found, at);
          remaining = __shfl_sync(0xffffffffu, rank, at);
          cls = __shfl_sync(0xffffffffu, cls, at);
        }
      }
      meet();
      if (W > 1) { found = s_pick[rr][0]; remaining = (int)s_pick[rr][1]; cls = (int)s_pick[rr][2]; }
      // (The class ends at the largest key.  Without that limit lo + span would wrap where scores of both signs meet scores from 2^127
      // on, or infinities: key 0 would lie inside the class, and the test for keys above it would take nearly all of them.)
      span = min((1u << shift) - 1u, span - (found << shift));
      lo += found << shift;
      if (shift == 0) { T = lo; need_eq = remaining; n_eq = cls; break; }
      // A class of at most 32 keys (the usual case after one pass) is finished by rank: its keys are gathered, each lane of one
      // warp ranks one of them against the others.  The columns above the class are kept: their number is taken on the way.
      if (cls <= 32) {
        int kept = 0;
        for (int j = j_mine; j - 4 * lane < j_hi; j += 128) {
          const uint4 kq = *reinterpret_cast<const uint4*>(keys + j);
          const bool a0 = kq.x - lo <= span, a1 = kq.y - lo <= span, a2 = kq.z - lo <= span, a3 = kq.w - lo <= span;
          if (W > 1) kept += (kq.x > lo + span) + (kq.y > lo + span) + (kq.z > lo + span) + (kq.w > lo + span);
          if (a0 | a1 | a2 | a3) {
            const int first = (int)atomicAdd(&s_found[rr], (uint32_t)a0 + (uint32_t)a1 + (uint32_t)a2 + (uint32_t)a3);
            int to = first;
            if (a0) s_list[rr][to++] = kq.x;
            if (a1) s_list[rr][to++] = kq.y;
            if (a2) s_list[rr][to++] = kq.z;
            if (a3) s_list[rr][to++] = kq.w;
            if (W > 1) for (int q = first; q < to; ++q) s_own[rr][q] = (uint32_t)w;
          }
        }
        if (W > 1) {
          kept = (int)__reduce_add_sync(0xffffffffu, (uint32_t)kept);
          if (lane == 0) s_cnt[rr][0][w] = kept;
        }
        meet();
        if (W == 1 || w == 0) {
          const uint32_t x = lane < cls ? s_list[rr][lane] : 0u;
          int G = 0, E = 0;                              // keys of the class larger than / equal to this lane's
#pragma unroll 4
          for (int l = 0; l < cls; ++l) {
            const uint32_t y = __shfl_sync(0xffffffffu, x, l);
            G += y > x; E += y == x;
          }
          const int ts = __ffs(__ballot_sync(0xffffffffu, x != 0u && G < remaining && remaining <= G + E)) - 1;
          T = __shfl_sync(0xffffffffu, x, ts);
          need_eq = remaining - __shfl_sync(0xffffffffu, G, ts);
          n_eq = __shfl_sync(0xffffffffu, E, ts);
          if (W > 1) {
            const uint32_t own = lane < cls ? s_own[rr][lane] : 0xffffffffu;
            int add = 0;
#pragma unroll
            for (int q = 0; q < W; ++q) { const int more = __popc(__ballot_sync(0xffffffffu, own == (uint32_t)q && x >= T)); if (lane == q) add = more; }
            if (lane < W) s_cnt[rr][0][lane] += add;
            if (lane == 0) { s_pick[rr][0] = T; s_pick[rr][1] = (uint32_t)need_eq; s_pick[rr][2] = (uint32_t)n_eq; }
          }
        }
        if (W > 1) {
          meet();
          T = s_pick[rr][0]; need_eq = (int)s_pick[rr][1]; n_eq = (int)s_pick[rr][2];
          counted = true;
        }
        break;
      }
      shift = max(shift - 8, 0);
      if (W == 1) { clear_hist(); meet(); }
    }
  }
  // ---- the list: kept columns in ascending order.  A warp's columns follow those of the warps before it.
  auto publish = [&](int which, uint32_t limit, bool equal) {   // a warp's columns with key >= limit, or == limit
    int cnt = 0;
    for (int j = j_mine; j - 4 * lane < j_hi; j += 128) {
      const uint4 kq = *reinterpret_cast<const uint4*>(keys + j);
      cnt += (equal ? kq.x == limit : kq.x >= limit) + (equal ? kq.y == limit : kq.y >= limit) + (equal ? kq.z == limit : kq.z >= limit) +
             (equal ? kq.w == limit : kq.w >= limit);
    }
    cnt = (int)__reduce_add_sync(0xffffffffu, (uint32_t)cnt);
    if (lane == 0) s_cnt[rr][which][w] = cnt;
    meet();
  };
  auto before = [&](int which) -> int {                  // columns of the warps before this one
    int x = 0;
    if (W > 1) for (int q = 0; q < w; ++q) x += s_cnt[rr][which][q];
    return x;
  };
  if (need_eq < n_eq) {              // ties at T that are not all kept: the later ones are struck out (rare)
    if (W > 1) publish(1, T, true);
    int rank0 = before(1);
    for (int j = j_mine; j - 4 * lane < j_hi; j += 128) {
      uint32_t* at = keys + j;
      int cnt = 0, rank = rank0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t bal = __ballot_sync(0xffffffffu, at[u] == T);
        cnt += __popc(bal); rank += __popc(bal & lt_mask);
      }
      rank0 += cnt;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (at[u] == T) { if (rank >= need_eq) at[u] = 0u; ++rank; }
    }
    counted = W == 1;
  }
  if (!counted) publish(0, T, false);
  int run = (sink_f ? 1 : 0) + before(0);
  for (int j = j_mine; j - 4 * lane < j_hi; j += 128) {
    const uint4 kq = *reinterpret_cast<const uint4*>(keys + j);
    const uint32_t b0 = __ballot_sync(0xffffffffu, kq.x >= T), b1 = __ballot_sync(0xffffffffu, kq.y >= T);
    const uint32_t b2 = __ballot_sync(0xffffffffu, kq.z >= T), b3 = __ballot_sync(0xffffffffu, kq.w >= T);
    int at = run + __popc(b0 & lt_mask) + __popc(b1 & lt_mask) + __popc(b2 & lt_mask) + __popc(b3 & lt_mask);
    run += __popc(b0) + __popc(b1) + __popc(b2) + __popc(b3);
    if (kq.x >= T) out[at++] = j;
    if (kq.y >= T) out[at++] = j + 1;
    if (kq.z >= T) out[at++] = j + 2;
    if (kq.w >= T) out[at] = j + 3;
  }
  if (w == 0 && lane == 0) {
    if (sink_f) out[0] = 0;
    if (diag_f) out[out1 - out0 - 1] = ri.i;
  }
}

// Threshold lists, and TopK lists of rows beyond kTopkRowMax: a warp per row.
__global__ void __launch_bounds__(kMaskWarps * 32)
fill_kernel(SeqMeta m, RowBand band, const float* scores, seer_mask_params p, const int32_t* row_ptr,
            int32_t* col_idx, int64_t col_capacity) {
  __shared__ __align__(16) uint32_t hist_smem[kMaskWarps * 256];      // 256 bins per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r = band.row_lo + (int64_t)blockIdx.x * kMaskWarps + warp;
  const RowInfo ri = decode_row(m, band, scores, r);
  grid_wait();
  if (!ri.valid || ri.skip) return;
  const int n = ri.i + 1;
  const int32_t out0 = row_ptr[r], out1 = row_ptr[r + 1];
  if ((int64_t)out1 > col_capacity) return;   // this row (and all later ones) do not fit; status already raised
  int32_t* out = col_idx + out0;
  const uint32_t lt_mask = (1u << lane) - 1u;

  if (ri.i >= ri.nb - p.dense_tail_blocks) {           // a dense row at the end of the sequence: every causal block
    for (int j = lane; j < n; j += 32) out[j] = j;
    return;
  }
  if (p.mode == SEER_THRESHOLD) {
    int written = 0;
    int head = 0;
    if ((reinterpret_cast<uintptr_t>(ri.s) & 15) == 0) {
      // four consecutive columns per lane: the lane's kept columns follow those of the lanes below it
      head = n & ~127;
      for (int base = 0; base < head; base += 128) {
        const int j = base + 4 * lane;
        const float4 v = *reinterpret_cast<const float4*>(ri.s + j);
        const bool k0 = is_forced(j, ri.i, p.flags) || v.x > p.threshold, k1 = is_forced(j + 1, ri.i, p.flags) || v.y > p.threshold;
        const bool k2 = is_forced(j + 2, ri.i, p.flags) || v.z > p.threshold, k3 = is_forced(j + 3, ri.i, p.flags) || v.w > p.threshold;
        const int mine = (int)k0 + (int)k1 + (int)k2 + (int)k3;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += u;
        }
        int at = written + incl - mine;
        if (k0) out[at++] = j;
        if (k1) out[at++] = j + 1;
        if (k2) out[at++] = j + 2;
        if (k3) out[at++] = j + 3;
        written += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    for (int base = head; base < n; base += 32) {
      const int j = base + lane;
      const bool keep = j < n && (is_forced(j, ri.i, p.flags) || ri.s[j] > p.threshold);
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      if (keep) out[written + __popc(bal & lt_mask)] = j;
      written += __popc(bal);
    }
    return;
  }

  // ---- TopK
  const int nf = num_forced(ri.i, p.flags);
  const int take = max(keep_count(n, p) - nf, 0);
  auto key_at = [&](int j) -> uint32_t {
    return is_forced(j, ri.i, p.flags) ? 0u : score_key(ri.s[j]);
  };
  int c = 0;
  uint32_t k_and = 0xffffffffu, k_or = 0u;     // over the candidates' keys: the bits all of them share are k_and | ~k_or
#pragma unroll 4
  for (int j = lane; j < n; j += 32) {
    const uint32_t kk = key_at(j);
    c += kk != 0u;
    k_or |= kk;
    k_and &= kk != 0u ? kk : 0xffffffffu;
  }
  const int ncand = warp_sum(c);
  k_and = __reduce_and_sync(0xffffffffu, k_and);
  k_or = __reduce_or_sync(0xffffffffu, k_or);

  uint32_t T = 0u;      // key of the last kept candidate; kept: key > T, plus the first need_eq with key == T
  int need_eq = 0;
  if (take >= ncand) {
    T = 0u; need_eq = 0;            // every candidate is kept (key >= 1 > 0)
  } else if (take == 0) {
    T = 0xffffffffu; need_eq = 0;   // nothing beyond the forced blocks
  } else {
    // radix select, up to 8 bits a pass from the top, the scores re-read in every pass: a histogram of the current digit of the keys
    // that match the prefix found so far, walked from the largest digit down.  The leading bits that all keys share need no pass.
    uint32_t* hist = hist_smem + warp * 256;
    const uint32_t differ = k_and ^ k_or;                                 // bit set: not all keys agree there
    int hi_bit = differ == 0u ? 0 : 31 - __clz(differ);                   // highest differing bit
    uint32_t prefix_mask = hi_bit >= 31 ? 0u : ~((2u << hi_bit) - 1u);    // the shared leading bits
    uint32_t prefix = k_or & prefix_mask;
    int remaining = take;           // rank (1-based, from the top) still to locate inside the current prefix class
    for (int top = hi_bit; top >= 0; top -= 8) {                          // this pass: bits top .. max(top - 7, 0)
      const int shift = max(top - 7, 0);
      const uint32_t dmask = (2u << (top - shift)) - 1u;
      for (int b = lane; b < 256; b += 32) hist[b] = 0u;
      __syncwarp();
      for (int j = lane; j < n; j += 32) {
        const uint32_t kk = key_at(j);
        if (kk != 0u && (kk & prefix_mask) == prefix) atomicAdd(&hist[(kk >> shift) & dmask], 1u);
      }
      __syncwarp();
      // lane l owns digits 8l .. 8l+7; suffix sums over lanes give the number of keys with a larger digit
      uint32_t c[8], lane_total = 0u;
      {
        const uint4 h0 = *reinterpret_cast<const uint4*>(hist + lane * 8), h1 = *reinterpret_cast<const uint4*>(hist + lane * 8 + 4);
        c[0] = h0.x; c[1] = h0.y; c[2] = h0.z; c[3] = h0.w; c[4] = h1.x; c[5] = h1.y; c[6] = h1.z; c[7] = h1.w;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) lane_total += c[e];
      uint32_t above = lane_total;                       // inclusive suffix sum over lanes >= this lane
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(0xffffffffu, above, o);
        if (lane + o < 32) above += v;
      }
      above -= lane_total;                               // keys in lanes with larger digits
      // the digit holding rank `remaining` lies in the lane where above < remaining <= above + lane_total
      const bool mine = (int)above < remaining && remaining <= (int)(above + lane_total);
      uint32_t digit = 0u; int new_remaining = 0;
      if (mine) {
        uint32_t acc = above;
#pragma unroll
        for (int e = 7; e >= 0; --e) {
          if ((int)acc < remaining && remaining <= (int)(acc + c[e])) { digit = (uint32_t)(lane * 8 + e); new_remaining = remaining - (int)acc; }
          acc += c[e];
        }
      }
      const uint32_t owner = __ballot_sync(0xffffffffu, mine);
      const int src = __ffs(owner) - 1;
      digit = __shfl_sync(0xffffffffu, digit, src);
      remaining = __shfl_sync(0xffffffffu, new_remaining, src);
      prefix |= digit << shift;
      prefix_mask |= dmask << shift;
      __syncwarp();
    }
    T = prefix;                      // the take-th largest key; `remaining` of the keys equal to it are kept
    need_eq = remaining;
  }
  int written = 0, eq_seen = 0;
  for (int base = 0; base < n; base += 32) {
    const int j = base + lane;
    const uint32_t kk = j < n ? key_at(j) : 0u;
    const bool forced = j < n && is_forced(j, ri.i, p.flags);
    const bool eq = kk != 0u && kk == T;
    const uint32_t eq_bal = __ballot_sync(0xffffffffu, eq);
    const bool keep = forced || (kk != 0u && kk > T) || (eq && eq_seen + __popc(eq_bal & lt_mask) < need_eq);
    const uint32_t bal = __ballot_sync(0xffffffffu, keep);
    if (keep) out[written + __popc(bal & lt_mask)] = j;
    written += __popc(bal);
    eq_seen += __popc(eq_bal);
  }
}

template <int W>
static cudaError_t launch_topk_w(const SeqMeta& m, const RowBand& band, const float* scores, const float2* stats, bool logits, const seer_mask_params& p,
                                 const int32_t* row_ptr, int32_t* col_idx, int64_t col_capacity, cudaStream_t stream) {
  constexpr int kRows = W == 1 ? 4 : 1, kThreads = W == 1 ? 128 : W * 32;
  const int cap = (m.max_nb + 128 * W - 1) / (128 * W) * (128 * W);
  return launch_next(logits ? topk_kernel<W, true> : topk_kernel<W, false>, (unsigned)((band.row_hi - band.row_lo + kRows - 1) / kRows), kThreads, (size_t)kRows * cap * 4,
                     stream, m, band, scores, stats, p, row_ptr, col_idx, col_capacity, cap);
}
// At most 2048 keys per warp (4096-block rows: two warps 4 % slower than four); kTopkRowMax = 8 warps' worth.  `logits`: the scores'
// place holds logits (launch_gate_logits_band), `stats` their statistics.
static cudaError_t launch_topk(const SeqMeta& m, const RowBand& band, const float* scores, const float2* stats, bool logits, const seer_mask_params& p,
                               const int32_t* row_ptr, int32_t* col_idx, int64_t col_capacity, cudaStream_t stream) {
  if (m.max_nb <= 2048) return launch_topk_w<1>(m, band, scores, stats, logits, p, row_ptr, col_idx, col_capacity, stream);
  if (m.max_nb <= 8192) return launch_topk_w<4>(m, band, scores, stats, logits, p, row_ptr, col_idx, col_capacity, stream);
  return launch_topk_w<8>(m, band, scores, stats, logits, p, row_ptr, col_idx, col_capacity, stream);
}

bool mask_takes_logits(const SeqMeta& m, const seer_mask_params& p) { return p.mode != SEER_THRESHOLD && m.max_nb <= kTopkRowMax; }

int launch_mask_band(seer_ctx* ctx, const SeqMeta& m, const float* scores, const float2* stats, bool logits, const ScoreBand& sb, int64_t row_lo,
                     int64_t row_hi, bool first, const seer_mask_params& p, int32_t* row_ptr, int32_t* col_idx,
                     int64_t col_capacity, int64_t* nnz_out, cudaStream_t stream) {
  if (row_hi <= row_lo) return 0;
  const RowBand band = {row_lo, row_hi, sb};
  const unsigned grid = (unsigned)((row_hi - row_lo + kMaskWarps - 1) / kMaskWarps);
  const bool from_stats = stats != nullptr && p.mode != SEER_THRESHOLD, small = !from_stats && small_mask(row_hi - row_lo, m.max_nb, p.mode);
  cudaError_t e = small
      ? launch_next(count_scan_kernel, 1, 1024, 0, stream, m, band, scores, p, row_ptr, first ? 1 : 0, col_capacity, nnz_out, ctx->d_status)
      : from_stats
      ? launch_next(logits ? topk_count_kernel<true> : topk_count_kernel<false>, (unsigned)((row_hi - row_lo + 31) / 32), 128, 0, stream, m, band, scores, stats, p, row_ptr)
      : launch_next(count_kernel, grid, kMaskWarps * 32, 0, stream, m, band, scores, p, row_ptr);
  if (e == cudaSuccess && !small) e = launch_scan(row_hi - row_lo, row_ptr + row_lo, first ? 1 : 0, col_capacity, nnz_out, ctx->d_status, stream);
  if (e == cudaSuccess)
    e = p.mode != SEER_THRESHOLD && m.max_nb <= kTopkRowMax
        ? launch_topk(m, band, scores, stats, logits, p, row_ptr, col_idx, col_capacity, stream)
        : launch_next(fill_kernel, grid, kMaskWarps * 32, 0, stream, m, band, scores, p, row_ptr, col_idx, col_capacity);
  return e == cudaSuccess ? (small ? 2 : 3) : -(int)e;
}

int launch_mask(seer_ctx* ctx, const SeqMeta& m, const float* scores, const seer_mask_params& p, int32_t* row_ptr,
                int32_t* col_idx, int64_t col_capacity, int64_t* nnz_out, cudaStream_t stream) {
  if (m.rows == 0) {
    cudaMemsetAsync(row_ptr, 0, sizeof(int32_t), stream);
    if (nnz_out) cudaMemsetAsync(nnz_out, 0, sizeof(int64_t), stream);
    return 0;
  }
  const ScoreBand all = {0, m.total_blocks, 0, m.num_q_heads, 0, 0, 0};
  return launch_mask_band(ctx, m, scores, nullptr, false, all, 0, m.rows, true, p, row_ptr, col_idx, col_capacity, nnz_out, stream);
}

// ----------------------------------------------------------------------------------------------- 128-token lists -> 64-token lists
// A 128-token block j is the pair of 64-token blocks (2j, 2j + 1); the query rows of 128-token block i are the 64-token
// rows 2i and 2i + 1.  Causality inside the diagonal block: row 2i sees 2i only, row 2i + 1 sees 2i and 2i + 1.  Every
// other listed block j < i contributes both halves to both rows (they exist: only a sequence's last block can be
// shorter than 65 tokens).  An entry j > i is not causal; it is passed on as (2j, 2j + 1) and the attention call
// reports it.  One warp per 64-token row; `fill` = false counts, true writes.
template <bool kFill>
__global__ void __launch_bounds__(kMaskWarps * 32)
expand_kernel(SeqMeta m128, SeqMeta m64, const int32_t* row_ptr128, const int32_t* col_idx128,
              int32_t* row_ptr64, int32_t* col_idx64, int64_t col_capacity64) {
  grid_wait();
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * kMaskWarps + (threadIdx.x >> 5);
  if (r >= m64.rows) return;
  const int b = find_sequence(m64.blk_off, m64.batch, (int)(r / m64.num_q_heads));
  const int nb64 = m64.blk_off[b + 1] - m64.blk_off[b], nb128 = m128.blk_off[b + 1] - m128.blk_off[b];
  const int64_t local = r - (int64_t)m64.num_q_heads * m64.blk_off[b];
  const int h = (int)(local / nb64);
  const int i64 = (int)(local - (int64_t)h * nb64);
  const int i128 = i64 >> 1;
  const bool odd = (i64 & 1) != 0;
  const int64_t src = (int64_t)m128.num_q_heads * m128.blk_off[b] + (int64_t)h * nb128 + i128;
  const int32_t s0 = row_ptr128[src], s1 = row_ptr128[src + 1];
  uint32_t out0 = 0;
  if (kFill) {
    out0 = (uint32_t)row_ptr64[r];
    if ((int64_t)(uint32_t)row_ptr64[r + 1] > col_capacity64) return;    // does not fit; status already raised by the scan
  }
  int written = 0;
  for (int base = s0; base < s1; base += 32) {
    const int e = base + lane;
    const int j = e < s1 ? col_idx128[e] : -1;
    const int c = e < s1 ? ((j == i128 && !odd) ? 1 : 2) : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (kFill && c > 0) {
      int32_t* dst = col_idx64 + (size_t)out0 + written + incl - c;
      dst[0] = 2 * j;
      if (c == 2) dst[1] = 2 * j + 1;
    }
    written += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (!kFill && lane == 0) row_ptr64[r + 1] = written;
}

int launch_expand_lists(seer_ctx* ctx, const SeqMeta& m128, const SeqMeta& m64, const int32_t* row_ptr128,
                        const int32_t* col_idx128, int32_t* row_ptr64, int32_t* col_idx64, int64_t col_capacity64,
                        int64_t* nnz_out, cudaStream_t stream) {
  if (m64.rows == 0) {
    cudaMemsetAsync(row_ptr64, 0, sizeof(int32_t), stream);
    if (nnz_out) cudaMemsetAsync(nnz_out, 0, sizeof(int64_t), stream);
    return 0;
  }
  const unsigned grid = (unsigned)((m64.rows + kMaskWarps - 1) / kMaskWarps);
  cudaError_t e = launch_next(expand_kernel<false>, grid, kMaskWarps * 32, 0, stream, m128, m64, row_ptr128, col_idx128, row_ptr64, col_idx64, col_capacity64);
  if (e == cudaSuccess) e = launch_scan(m64.rows, row_ptr64, 1, col_capacity64, nnz_out, ctx->d_status, stream);
  if (e == cudaSuccess)
    e = launch_next(expand_kernel<true>, grid, kMaskWarps * 32, 0, stream, m128, m64, row_ptr128, col_idx128, row_ptr64, col_idx64, col_capacity64);
  return e == cudaSuccess ? 3 : -(int)e;
}

seer_status init_mask(seer_ctx* ctx) {
  (void)ctx;
  const bool ok = cudaFuncSetAttribute(topk_kernel<8, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTopkRowMax * 4) == cudaSuccess &&
                  cudaFuncSetAttribute(topk_kernel<8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTopkRowMax * 4) == cudaSuccess;
  return ok ? SEER_OK : SEER_ERR_CUDA;
}

}  // namespace seer
