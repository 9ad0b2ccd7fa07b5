// The largest probability of every listed 64 x 64 tile (Sec. 3.2, Eq. 2 on the listed blocks) for a CTA all of whose pairs of query blocks have one list
// each: the pipeline of attn_pair.cu without V, its tensor memory four S buffers and its K ring five tiles deep.  A tile's K, 32 KB, serves
// four blocks; the maxima are attn_tc_kernel's bit for bit.  16 384 tokens, 32 heads, all blocks: 1146 -> 797 us (a
// kernel of its own, 384 threads: 797), the tensor pipe 94 % active with its operands' reads.  (Q from tensor memory, which halves what the MMAs read of shared memory, and two tiles
// at a time in a group: no gain.)
#pragma once

#include "attn_pair.cuh"

namespace seer {
namespace tp {

// Whether all pairs dealt to this CTA have one list each: pair by pair of its 16 warps; where lists differ the first sixteen say so.  (Whole CTA.)
template <bool kChunk>
__device__ __forceinline__ bool share_agrees(const SeqMeta& m, const int32_t* row_ptr, const int32_t* col_idx, int warp, int lane) {
  for (uint32_t k = 0; k == 0 || (int64_t)k * gridDim.x < m.pair_units; k += 16) {
    const int64_t w = dealt_pair(m, k + (uint32_t)warp);
    const bool ok = w < 0 || pair_ok<kChunk, true>(m, row_ptr, reinterpret_cast<const uint32_t*>(col_idx), w, lane);
    if (__syncthreads_or(!ok)) return false;
  }
  return true;
}

constexpr uint32_t kMaxKUnits = 5, kMaxS = 4;
// behind the K ring: the maxima that two warps exchange, then barriers and item slots, in the room that attn_tc_kernel has for its own
constexpr uint32_t kOffMaxima = kOffK + kMaxKUnits * kUnit, kOffMaxBar = kOffMaxima + 1024, kOffMaxRing = kOffMaxBar + 256, kMaxEnd = kOffMaxRing + 4 * 64;
enum MaxBar { M_Q_FULL = 0 /* + buf */, M_Q_EMPTY = 2, M_K_FULL = 4 /* + unit */, M_K_EMPTY = 9, M_S_FULL = 14 /* + buf */, M_TAKEN = 18, M_ITEM_FULL = 22 /* + slot */, M_ITEM_EMPTY = 26, kMaxBars = 30 };
static_assert(kMaxBars <= 32, "barriers of the block maxima");
__device__ __forceinline__ void max_init(uint32_t base, int i) {   // (by a warp, a barrier each)
  if (i < kMaxBars) mbar_init(base + kOffMaxBar + 8u * (uint32_t)i, i >= M_TAKEN && i < M_TAKEN + (int)kMaxS ? 8 : i >= M_ITEM_EMPTY && i < M_ITEM_EMPTY + 4 ? 9 : 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ uint32_t max_ring(const Shared& sh, uint32_t n) { return sh.base + kOffMaxRing + (n & 3u) * 64u; }

// The roles of a CTA of 16 warps: warp 0 producer of Q and K, warp 1 MMA issuer, warps 4-7 and 8-11 the maxima of the even and the odd list positions.
template <bool kChunk, int kHelpers, int kGroups>
__device__ __forceinline__ void block_max_pairs(const CUtensorMap& map_q, const CUtensorMap& map_k, const SeqMeta& m, Shared sh, unsigned char* smem, uint32_t tmem, int warp, int lane,
                                                const int32_t* row_ptr, const int32_t* col_idx, const float* lse, int* status, float* block_max) {
  sh.bar0 = sh.base + kOffMaxBar;
  if (warp < 4 || warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kHelpers));
    // ========================================================================================== producer of Q and K (TMA)
    if (warp == 0) {
      if (elect_one()) {
        const uint32_t* col = reinterpret_cast<const uint32_t*>(col_idx);
        uint32_t nitem = 0, ku = 0, kph = 0, cnt = 0;
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
          const int64_t w = dealt_pair(m, n);
          PairItem it{};
          if (w >= 0) it = decode_pair<kChunk, true>(m, row_ptr, w);
          const int tiles = (it.len + 1) >> 1, g = it.h / m.group;
          const int x0 = it.n[0] > 0 ? (int)ld_global(col + it.l0 + it.n[0] - 1) : -1, x1 = it.n[1] > 0 ? (int)ld_global(col + it.l0 + it.n[1] - 1) : -1;
          if (!mbar_wait(sh, M_ITEM_EMPTY + (int)(n & 3u), ((n >> 2) & 1u) ^ 1u, status)) break;
          st_shared_v4(max_ring(sh, n), (uint32_t)it.h, (uint32_t)it.tok0, (uint32_t)it.l[0], w >= 0 ? (uint32_t)it.len : 0xffffffffu);
          st_shared_v4(max_ring(sh, n) + 16u, (uint32_t)it.l[1], (uint32_t)it.n[0], (uint32_t)it.n[1], (uint32_t)it.valid[0] | (uint32_t)it.valid[1] << 16);
          st_shared_v4(max_ring(sh, n) + 32u, (uint32_t)(it.n[0] - (x0 == it.i0)), (uint32_t)(it.n[1] - (x1 == it.i0 + 1)), 0u, 0u);
          mbar_arrive(sh.bar(M_ITEM_FULL + (int)(n & 3u)));
          if (w < 0) break;
          if (tiles == 0) continue;
          int ja = (int)ld_global(col + it.l0), jb = it.len > 1 ? (int)ld_global(col + it.l0 + 1) : -1;
          const uint32_t qb = nitem & 1u, qf = sh.bar(M_Q_FULL + (int)qb);
          if (!mbar_wait(sh, M_Q_EMPTY + (int)qb, ((nitem >> 1) & 1u) ^ 1u, status)) break;
          mbar_expect_tx(qf, it.valid[0] > 0 && it.valid[1] > 0 ? kQBytes : kQBytes / 2);
#pragma unroll
          for (int half = 0; half < 2; ++half)
            if (it.valid[half] > 0)
#pragma unroll
              for (int dh = 0; dh < 2; ++dh)
                tma_load_3d(sh.base + kOffQ + qb * kQBytes + (uint32_t)(2 * dh + half) * kHalfTile, &map_q, qf, 64 * dh, it.h, it.tok0 + 64 * half);
          ++nitem;
          for (int t = 0; t < tiles; ++t, ++cnt) {
            const int p = 2 * t + 2;
            const int ra = p < it.len ? (int)ld_global(col + it.l0 + p) : -1, rb = p + 1 < it.len ? (int)ld_global(col + it.l0 + p + 1) : -1;   // next pair
            const bool has_b = jb >= 0;
            const int ta = it.s0 + ja * kBlock, tb = it.s0 + jb * kBlock;
            if (!mbar_wait(sh, M_K_EMPTY + (int)ku, kph ^ 1u, status)) { ok = false; break; }
            const uint32_t fb = sh.bar(M_K_FULL + (int)ku), dst = sh.base + kOffK + ku * kUnit;
            // test hook: one K copy that is never issued, so that the issuer's wait for it runs out
            if (blockIdx.x != 0 || m.lose_v_copy < 0 || cnt != (uint32_t)m.lose_v_copy) {
              mbar_expect_tx(fb, has_b ? kUnit : kUnit / 2);
#pragma unroll
              for (int dh = 0; dh < 2; ++dh) {
                tma_load_3d(dst + (uint32_t)dh * 2 * kHalfTile, &map_k, fb, 64 * dh, g, ta);
                if (has_b) tma_load_3d(dst + (uint32_t)dh * 2 * kHalfTile + kHalfTile, &map_k, fb, 64 * dh, g, tb);
              }
            }
            if (++ku == kMaxKUnits) { ku = 0; kph ^= 1u; }
            ja = ra; jb = rb;
          }
        }
      }
    }
    // ========================================================================================== MMA issuer
    else if (warp == 1) {
      if (elect_one()) {
        const uint64_t hi = make_desc(0, 16, 1024) & 0xffffffff00000000ull;
        const uint32_t kd_lo = (uint32_t)make_desc(sh.base + kOffK, 16, 1024), qd_lo = (uint32_t)make_desc(sh.base + kOffQ, 16, 1024);
        uint32_t cs = 0, ku = 0, kph = 0, nitem = 0;         // tiles issued, ring position, items with tiles
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
          if (!mbar_wait(sh, M_ITEM_FULL + (int)(n & 3u), (n >> 2) & 1u, status)) break;
          const int len = (int)ld_shared_u32(max_ring(sh, n) + 12u);
          mbar_arrive(sh.bar(M_ITEM_EMPTY + (int)(n & 3u)));
          if (len < 0) break;
          if (len == 0) continue;
          const uint32_t qlo = qd_lo + (nitem & 1u) * (kQBytes >> 4);
          if (!mbar_wait(sh, M_Q_FULL + (int)(nitem & 1u), (nitem >> 1) & 1u, status)) break;
          for (int t = (len + 1) >> 1; t > 0; --t, ++cs) {
            // the groups have taken the maxima of this S buffer's previous tile
            if (!mbar_wait(sh, M_TAKEN + (int)(cs & 3u), ((cs >> 2) & 1u) ^ 1u, status)) { ok = false; break; }
            if (!mbar_wait(sh, M_K_FULL + (int)ku, kph, status)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem + (cs & 3u) * 128u, klo = kd_lo + ku * (kUnit >> 4);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t off = (uint32_t)((kk >> 2) * (2 * kHalfTile >> 4) + (kk & 3) * 2);
              tc_mma_ss(d, hi | (uint64_t)(qlo + off), hi | (uint64_t)(klo + off), kIdescS, kk != 0 ? 1u : 0u);
            }
            tc_commit(sh.bar(M_S_FULL + (int)(cs & 3u)));
            tc_commit(sh.bar(M_K_EMPTY + (int)ku));
            if (++ku == kMaxKUnits) { ku = 0; kph ^= 1u; }
          }
          if (!ok) break;
          tc_commit(sh.bar(M_Q_EMPTY + (int)(nitem & 1u)));
          ++nitem;
        }
      }
    }
  }
  // ============================================================================================ maxima: a thread per row and list parity
  else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGroups));
    const int g = (warp - 4) >> 2, quad = warp & 3, half = quad >> 1;
    const int r = quad * 32 + lane, row = r & 63;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const float sl2 = m.softmax_scale * 1.4426950408889634f;
    const int64_t lse_stride = kChunk ? m.total_q_tokens : m.total_tokens;
    int* other = reinterpret_cast<int*>(smem + kOffMaxima) + (2 * g + half) * 64;   // [2][32]: the second warp's maxima of 32 tiles
    const int bar_block = 1 + 2 * g + half;                 // the two warps of a query block
    constexpr int bar_vote = 5, kBoth = 256;
    uint32_t cnt = 0, flushes = 0;
    bool lost = false;                                      // this warp, or its neighbour, has given up
    for (uint32_t n = 0;; ++n) {
      bool fail = lost || !mbar_wait_warp(sh, M_ITEM_FULL + (int)(n & 3u), (n >> 2) & 1u, status);
      uint4 a{}, b{}, c{};
      if (!fail) { a = ld_shared_v4(max_ring(sh, n)); b = ld_shared_v4(max_ring(sh, n) + 16u); c = ld_shared_v4(max_ring(sh, n) + 32u); }
      __syncwarp();
      if (lane == 0 && !fail) mbar_arrive(sh.bar(M_ITEM_EMPTY + (int)(n & 3u)));
      const int len = (int)a.w;
      // A warp with an item waits in it for its neighbour: so either all warps have the item, or none goes on.
      if (named_bar_or(bar_vote, kBoth, fail) || len < 0) break;
      const int mine_n = (int)(half ? b.z : b.y), plain = (int)(half ? c.y : c.x), l0 = (int)(half ? b.x : a.z);
      const int valid = (int)(half ? b.w >> 16 : b.w & 0xffffu);
      float L = row < valid ? lse[(int64_t)a.x * lse_stride + (int)a.y + 64 * half + row] : 0.f;
      if (!(fabsf(L) < 3.0e38f)) L = 0.f;                   // a query without a key has no probabilities to report
      const float L2 = L * 1.4426950408889634f;
      // Lane k holds the warp's maximum of the k-th tile since the block's two warps last met, as an order-preserving integer: they meet every
      // 32 tiles (every tile: 16k tokens, all blocks, 850 us where this takes 755).
      int key = 0, first_p = g;
      for (int p = g; p < len + g; p += 2, ++cnt) {         // (both groups take every tile, the second one without a block in an odd list's last)
        const uint32_t sbuf = cnt & 3u;
        fail = !mbar_wait_warp(sh, M_S_FULL + (int)sbuf, (cnt >> 2) & 1u, status);
        if (fail) break;
        tc_fence_after();
        const uint32_t s_addr = tmem + lane_addr + sbuf * 128u + (uint32_t)g * 64u;
        float mx = -CUDART_INF_F;
        if (p < mine_n) mx = p < plain ? row_max<false>(s_addr, 63) : row_max<true>(s_addr, row);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sh.bar(M_TAKEN + (int)sbuf));   // (this warp is done with the S buffer)
        if (row >= valid || !(mx == mx)) mx = -CUDART_INF_F;
        else mx = fmaf(mx, sl2, -L2);
        int k = __float_as_int(mx);
        k ^= (k >> 31) & 0x7fffffff;                        // order-preserving map float -> int
        k = __reduce_max_sync(0xffffffffu, k);
        const int at = (p - first_p) >> 1;
        if (lane == at) key = k;
        if (at == 31 || p + 2 >= len + g) {
          int* there = other + (flushes++ & 1u) * 32;
          if ((quad & 1) != 0) there[lane] = key;
          if (named_bar_or(bar_block, 64, false)) { lost = true; break; }
          const int mine = first_p + 2 * lane;
          if ((quad & 1) == 0 && lane <= at && mine < mine_n) {
            int kx = max(key, there[lane]);
            kx ^= (kx >> 31) & 0x7fffffff;
            block_max[l0 + mine] = exp2f(__int_as_float(kx));   // 2^(-inf) = 0: no causal pair
          }
          first_p = p + 2;
        }
      }
      if (fail) { named_bar_or(bar_block, 64, true); lost = true; }   // (the neighbour is waiting there, or will)
    }
  }
}

}  // namespace tp
}  // namespace seer
