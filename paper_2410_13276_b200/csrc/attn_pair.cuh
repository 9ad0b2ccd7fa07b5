// Pairs of query blocks (2u, 2u + 1) of a head and their lists: what the kernels that take them together, and those that leave them to these, share.
#pragma once

#include "attn_tc_common.cuh"

namespace seer {
namespace tp {

using namespace tcc;

constexpr uint32_t kHalfTile = 64 * 128;         // bytes of one d half of a 64-row tile (8 KB)
constexpr uint32_t kQBytes = 4 * kHalfTile;      // 32 KB: [d half][query block]
constexpr uint32_t kUnit = 4 * kHalfTile;        // a tile's K, [d half][block], or its V, [block][d half]
constexpr uint32_t kOffQ = 0, kOffK = 2 * kQBytes;   // two buffers of Q, then the rings
constexpr uint32_t kIdescS = make_idesc(false, false, 128u, 128u);

struct PairPlace {
  int h, i0, s0, tok0;         // first query block; first key token of the sequence; first row of block i0 in q / o / lse
  int valid[2];                // query rows of the two blocks (none: not there)
  int64_t row;                 // of block i0 in row_ptr
};
struct PairItem : PairPlace {
  int l0, len;                 // the longer list
  int l[2], n[2];              // both lists' starts and lengths
};

// The w-th pair: KV head by KV head of a sequence, from the last pair to the first, a pair's heads side by side.  kZigzag: every other KV head from the
// first pair to the last, so that the lists' lengths have no jump from one head to the next.
template <bool kChunk, bool kZigzag = false>
__device__ __forceinline__ PairPlace place_pair(const SeqMeta& m, int64_t w) {
  PairPlace it;
  const int p = find_sequence(m.pair_off, m.batch, (int)(w / m.num_q_heads)), before = m.pair_off[p];
  const int4 s = m.place[p];
  const int nb = (s.y + kBlock - 1) / kBlock, np = m.pair_off[p + 1] - before;
  const int first = kChunk ? nb - (m.qblk_off[p + 1] - m.qblk_off[p]) : 0;
  const int local = (int)(w - (int64_t)m.num_q_heads * before);
  const int g = local / (np * m.group);
  int rem = local - g * np * m.group;
  if (kZigzag && ((m.num_kv_heads - 1 - g) & 1)) rem = np * m.group - 1 - rem;
  it.i0 = 2 * ((nb + 1) / 2 - 1 - rem / m.group);
  it.h = g * m.group + rem % m.group;
  it.s0 = s.x;
  it.tok0 = s.x + it.i0 * kBlock + (kChunk ? s.w : 0);
  it.row = (int64_t)m.num_q_heads * s.z + (int64_t)it.h * nb + it.i0;
  it.valid[0] = it.i0 >= first ? min(kBlock, s.y - it.i0 * kBlock) : 0;
  it.valid[1] = it.i0 + 1 < nb ? min(kBlock, s.y - (it.i0 + 1) * kBlock) : 0;
  return it;
}
template <bool kChunk, bool kZigzag = false>
__device__ __forceinline__ PairItem decode_pair(const SeqMeta& m, const int32_t* row_ptr, int64_t w) {
  PairItem it;
  static_cast<PairPlace&>(it) = place_pair<kChunk, kZigzag>(m, w);
  const int l0 = row_ptr[it.row], l1 = row_ptr[it.row + 1], l2 = it.valid[1] > 0 ? row_ptr[it.row + 2] : l1;
  it.n[0] = it.valid[0] > 0 ? l1 - l0 : 0;
  it.n[1] = it.valid[1] > 0 ? l2 - l1 : 0;
  const bool second = it.n[1] >= it.n[0];
  it.l0 = second ? l1 : l0;
  it.len = second ? it.n[1] : it.n[0];
  it.l[0] = l0; it.l[1] = l1;
  return it;
}

// Whether the pair has one list: the same entries, all before the first block or, at the end of that block's list, the block itself; the second
// block may list one more, up to itself.  A pair's second block alone, or the first, where the other has no queries: entries before the
// block, the last one up to it.  (By a converged warp.)
template <bool kChunk, bool kZigzag = false>
__device__ __forceinline__ bool pair_ok(const SeqMeta& m, const int32_t* row_ptr, const uint32_t* col, int64_t w, int lane) {
  const PairItem it = decode_pair<kChunk, kZigzag>(m, row_ptr, w);
  const int l2 = it.n[1] >= it.n[0] ? it.l[0] : it.l[1];
  const bool both = it.valid[0] > 0 && it.valid[1] > 0;
  const int n = both ? min(it.n[0], it.n[1]) : 0;         // entries that both list
  const int own = it.valid[0] > 0 ? it.n[0] : it.n[1], top = it.valid[0] > 0 ? it.i0 : it.i0 + 1;   // the first block's list, or the only one
  bool ok = !both || it.n[1] == it.n[0] || it.n[1] == it.n[0] + 1;
  for (int b = 0; b < it.len && ok; b += 256) {           // (uniform in the warp)
    uint32_t x[8], y[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int p = b + 32 * e + lane;
      x[e] = p < it.len ? ld_global(col + it.l0 + p) : 0u;
      y[e] = p < n ? ld_global(col + l2 + p) : x[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int p = b + 32 * e + lane;
      ok = ok && x[e] == y[e] && (p >= it.len || x[e] < (uint32_t)(p < own - 1 ? top : p < own ? top + 1 : top + 2));
    }
    ok = __all_sync(0xffffffffu, ok);
  }
  return ok;
}

// The static deal of the block maxima: CTA c takes the pairs of every grid-sized round, from either end in turn.  In the zigzag order the longest
// share is 0.7 % above the mean for 16k tokens and 32 heads, all blocks (6 % with every head from its last pair on, 64 % for 9000 tokens).  -1: past the
// last one.
__device__ __forceinline__ int64_t dealt_pair(const SeqMeta& m, uint32_t k) {
  const int64_t w = (int64_t)k * gridDim.x + ((k & 1u) ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
  return w < m.pair_units ? w : -1;
}
// Whether all of a check's words are this call's (kPairWords of them at most, as many threads or more).
__device__ __forceinline__ bool lists_agree(const int* words, int nwords, int epoch) {
  return !__syncthreads_or((int)threadIdx.x < nwords && *(const volatile int*)(words + threadIdx.x) != epoch);
}

}  // namespace tp
}  // namespace seer
